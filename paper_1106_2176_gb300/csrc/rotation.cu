// Rotation-based M2L (the paper's GPU code rotates expansions so that the
// translation runs along z, O(p^3) per pair instead of O(p^4); Sec. 2.2 and
// the prior GPU work it cites).
//
// For a translation u = c_L - c_M, a rotation Q takes u to |u| z. In the
// rotated frame the irregular harmonics I_l^mu(|u| z) vanish unless mu = 0,
// where I_l^0 = l! / |u|^(l+1), so the translation couples only equal orders:
//   L'_n^m = (-1)^n sum_{j >= |m|} M'_j^-m (j+n)! / |u|^(j+n+1).
// M' (the multipoles seen from the rotated frame) and L (the locals back in
// the original frame) follow from M and L' by one dense map per degree n,
// (2n+1) x (2n+1) real on the packed coefficients: 2 sum_n (2n+1)^2 + O(p^3)
// multiply-adds per pair.
//
// The maps are built on the host in FP64. On the unit sphere both families
// are multiples of Yt_n^m = P_n^m(cos t) e^{i m f} sqrt((n-m)!/(n+m)!)
// (P without the Condon-Shortley phase): I_n^m = c_nm Yt_n^m and
// R_n^m = Yt_n^m / c_nm with c_nm = sqrt((n+|m|)! (n-|m|)!). A rotation acts
// unitarily on the Yt of one degree. With Q = R_y(-b) R_z(-a) (a, b the
// azimuth and polar angle of u), Yt^m(x) = e^{i m a} sum_m' V_mm'(b) Yt^m'(Qx)
// where V(b) is defined by Yt^m(R_y(b) y) = sum_m' V_mm'(b) Yt^m'(y). With
// this normalisation V_mm'(b) is the Wigner small-d matrix element
// d^n_{m'm}(b); it is evaluated in closed form from its Jacobi-polynomial
// expression (Edmonds, Angular Momentum in Quantum Mechanics, 1957, Eq.
// 4.1.23), once per distinct polar angle, and the azimuth enters as exact
// phases. Then, with U = diag(e^{i m a}) V:
//   M'^m' = sum_m M^m c_m U_mm' / c_m'        (multipoles into the frame)
//   L^m   = sum_m' L'^m' c_m U_mm' / c_m'     (locals back, U^-1 = U^H)

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <complex>
#include <exception>
#include <map>
#include <memory>
#include <mutex>
#include <thread>
#include <tuple>
#include <vector>

#include "fmm_internal.cuh"
#include "ptx_sm100.cuh"

namespace fmm {

using cplx = std::complex<double>;

// offset of degree n's (2n+1) x (2n+1) block in a per-vector map table
int rot_deg_off(int n) { return n * (4 * n * n - 1) / 3; }
int rot_map_size(int p) { return rot_deg_off(p); }

static double fact(int k)
{
    double f = 1;
    for (int i = 2; i <= k; i++) f *= i;
    return f;
}

static double binom(int n, int k) { return fact(n) / (fact(k) * fact(n - k)); }

// Jacobi polynomial P_k^(a,b)(x) by its three-term recurrence in the degree
// (Abramowitz & Stegun 22.7.1), stable for x in [-1, 1]
static double jacobi(int k, int a, int b, double x)
{
    if (k == 0) return 1.0;
    double p0 = 1.0, p1 = 0.5 * ((double)(a - b) + (double)(a + b + 2) * x);
    for (int j = 2; j <= k; j++) {
        const double s = (double)(2 * j + a + b);
        const double c1 = 2.0 * j * (double)(j + a + b) * (s - 2.0);
        const double c2 = (s - 1.0) * (double)(a * a - b * b);
        const double c3 = (s - 2.0) * (s - 1.0) * s;
        const double c4 = 2.0 * (double)(j + a - 1) * (double)(j + b - 1) * s;
        const double p2 = ((c2 + c3 * x) * p1 - c4 * p0) / c1;
        p0 = p1;
        p1 = p2;
    }
    return p1;
}

// Wigner small-d element d^n_{m'm}(b) from its Jacobi form: with
// k = min(n+m, n-m, n+m', n-m'), the exponents a = |m - m'|,
// c = |m + m'| (= 2n - 2k - a), and the sign (-1)^(m'-m) when m' > m,
//   d = sign sqrt(C(2n-k, k+a) / C(k+c, c)) sin(b/2)^a cos(b/2)^c P_k^(a,c)(cos b)
static double wigner_d(int n, int mp, int m, double b)
{
    const int k = std::min(std::min(n + m, n - m), std::min(n + mp, n - mp));
    int a, lam;
    if (k == n + m || k == n - mp) {
        a = mp - m;
        lam = mp - m;
    } else {
        a = m - mp;
        lam = 0;
    }
    const int c = 2 * n - 2 * k - a;
    const double sgn = (lam & 1) ? -1.0 : 1.0;
    return sgn * std::sqrt(binom(2 * n - k, k + a) / binom(k + c, c)) * std::pow(std::sin(0.5 * b), a) *
           std::pow(std::cos(0.5 * b), c) * jacobi(k, a, c, std::cos(b));
}

// V(b) for every degree n < p: Yt_n^m(R_y(b) y) = sum_m' V_mm' Yt_n^m'(y)
// with V_mm' = d^n_{m'm}(b). V[n] is (2n+1)^2 real, row m + n.
static std::vector<std::vector<double>> vmaps(int p, double b)
{
    std::vector<std::vector<double>> V(p);
    for (int n = 0; n < p; n++) {
        const int K = 2 * n + 1;
        V[n].resize((size_t)K * K);
        for (int m = -n; m <= n; m++)
            for (int mp = -n; mp <= n; mp++) V[n][(size_t)(m + n) * K + (mp + n)] = wigner_d(n, mp, m, b);
    }
    return V;
}

// real packed form of a complex degree-n map given as out^j = sum_i in^i T[i][j]
// (i, j = m + n): column b of the result is the map applied to packed basis vector b
static void packed(int n, const std::vector<cplx> &T, double *out)
{
    const int K = 2 * n + 1;
    std::vector<cplx> in(K), o(K);
    for (int b = 0; b < K; b++) {
        std::fill(in.begin(), in.end(), cplx(0, 0));
        const int m = (b + 1) / 2;
        const cplx e = b == 0 ? cplx(1, 0) : ((b & 1) ? cplx(1, 0) : cplx(0, 1));
        in[n + m] = e;
        if (m) in[n - m] = ((m & 1) ? -1.0 : 1.0) * std::conj(e);
        for (int j = 0; j < K; j++) {
            cplx s(0, 0);
            for (int i = 0; i < K; i++) s += in[i] * T[(size_t)i * K + j];
            o[j] = s;
        }
        out[0 * K + b] = o[n].real();
        for (int mm = 1; mm <= n; mm++) {
            out[(size_t)(2 * mm - 1) * K + b] = o[n + mm].real();
            out[(size_t)(2 * mm) * K + b] = o[n + mm].imag();
        }
    }
}

// V(b) cached per (p, b): the stencil has far fewer polar angles than vectors
static std::mutex g_v_mu;
static std::map<std::pair<int, double>, std::shared_ptr<const std::vector<std::vector<double>>>> g_v_cache;

static std::shared_ptr<const std::vector<std::vector<double>>> vmaps_cached(int p, double b)
{
    const auto key = std::make_pair(p, b);
    {
        std::lock_guard<std::mutex> lk(g_v_mu);
        auto it = g_v_cache.find(key);
        if (it != g_v_cache.end()) return it->second;
    }
    auto v = std::make_shared<const std::vector<std::vector<double>>>(vmaps(p, b));
    std::lock_guard<std::mutex> lk(g_v_mu);
    g_v_cache[key] = v;
    return v;
}

// forward (multipoles into the rotated frame) and backward (locals out of it)
// maps for translation u, each rot_map_size(p) doubles, degree blocks row-major
void rotation_maps(int p, const double u[3], double *A, double *B)
{
    const double rxy = std::hypot(u[0], u[1]);
    const double a = rxy > 0 ? std::atan2(u[1], u[0]) : 0.0, b = std::atan2(rxy, u[2]);
    auto V = vmaps_cached(p, b);
    for (int n = 0; n < p; n++) {
        const int K = 2 * n + 1;
        std::vector<cplx> T((size_t)K * K);
        for (int i = 0; i < K; i++) {
            const int m = i - n;
            const cplx ph = std::polar(1.0, m * a);
            const double cm = std::sqrt(fact(n + std::abs(m)) * fact(n - std::abs(m)));
            for (int j = 0; j < K; j++) {
                const int mp = j - n;
                const double cmp = std::sqrt(fact(n + std::abs(mp)) * fact(n - std::abs(mp)));
                T[(size_t)i * K + j] = cm * ph * (*V)[n][(size_t)i * K + j] / cmp;
            }
        }
        // both directions use T: M'^j = sum_i M^i T_ij, L^i = sum_j L'^j T_ij
        packed(n, T, A + rot_deg_off(n));
        std::vector<cplx> Tt((size_t)K * K);
        for (int i = 0; i < K; i++)
            for (int j = 0; j < K; j++) Tt[(size_t)j * K + i] = T[(size_t)i * K + j];
        packed(n, Tt, B + rot_deg_off(n));
    }
}

// the whole rotation M2L on the host, FP64, packed p^2 coefficients
void m2l_rotation_ref(int p, const double u[3], const double *M, double *L)
{
    const int PP = p * p;
    std::vector<double> A(rot_map_size(p)), B(rot_map_size(p)), Mr(PP), Lr(PP);
    rotation_maps(p, u, A.data(), B.data());
    for (int n = 0; n < p; n++) {
        const int K = 2 * n + 1;
        for (int r = 0; r < K; r++) {
            double s = 0;
            for (int c = 0; c < K; c++) s += A[rot_deg_off(n) + (size_t)r * K + c] * M[n * n + c];
            Mr[n * n + r] = s;
        }
    }
    const double d = std::sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    std::vector<double> g(2 * p);
    for (int l = 0; l < 2 * p - 1; l++) g[l] = fact(l) / std::pow(d, l + 1);
    for (int n = 0; n < p; n++)
        for (int m = 0; m <= n; m++) {
            double sr = 0, si = 0;
            for (int j = m; j < p; j++) {
                sr += Mr[re_idx(j, m)] * g[j + n];
                if (m) si += Mr[im_idx(j, m)] * g[j + n];
            }
            const double sg = ((n + m) & 1) ? -1.0 : 1.0;
            Lr[re_idx(n, m)] = sg * sr;
            if (m) Lr[im_idx(n, m)] = -sg * si;
        }
    for (int n = 0; n < p; n++) {
        const int K = 2 * n + 1;
        for (int r = 0; r < K; r++) {
            double s = 0;
            for (int c = 0; c < K; c++) s += B[rot_deg_off(n) + (size_t)r * K + c] * Lr[n * n + c];
            L[n * n + r] = s;
        }
    }
}

}  // namespace fmm

// ---------------------------------------------------------------------------
// device engine
//
// On the device the azimuth and the polar angle are applied apart. With the
// coefficients multiplied by c_nm, X^m = c_m M^m e^{ima} (a phase per order),
// and, because V is real and X^{-m} = (-1)^m conj(X^m), the polar rotation acts
// on real and imaginary parts separately:
//   Re M'^m' = sum_m T_mm' Re X^m / c_m',  T = V_mm' + (-1)^m V_{-m m'}  (X^0 halved)
//   Im M'^m' = sum_m Q_mm' Im X^m / c_m',  Q = V_mm' - (-1)^m V_{-m m'}
// two maps of (n+1)^2 and n^2 entries instead of one of (2n+1)^2. The way back
// takes the same two: L^m = c_m e^{ima} (sum_m' T_mm' Re L'^m' + i sum_m' Q_mm'
// Im L'^m') / c_m' (L'^0 halved), because (-1)^m' V_{m,-m'} = (-1)^m V_{-m,m'}.
// The maps T_mm' / c_m' and Q_mm' / c_m' depend on the polar angle alone: about
// 400 of them serve the 1,740 vectors of theta = 0.5.
//
// One CTA per tile of 32 target cells and range of the tile's vectors; lane i
// of every warp is target i, and the warps share the coefficients. Per vector:
//   gather   c M~ of the 32 sources (zero where absent), whole rows by cp.async,
//            transposed to [coefficient][target] in shared memory
//   forward  warps take (degree, part): e^{ima}, then a map row against the 32
//            targets at once, the map read by broadcast
//   along z  warps take (order, part): sums over the degrees of equal order
//   back     as forward
//   phases   e^{ima}, added to the warp's coefficients of L~ in registers
//            (FP32: TwoSum pairs)
// The (degree, part) jobs, K^2 multiply-adds each (K = n + 1 or n), are dealt
// to the warps by size. The next vector's rows and maps arrive while the
// current one is translated.
//
// Bound: FP32 by instruction issue (a map's 16 bytes are one load and two packed
// multiply-adds), FP64 by GB300's FP64 pipe. N = 60,001, p = 16, FP32: 7.9 ms;
// N = 50,000, p = 8, FP64: 18.2 ms. One warp per two targets with lanes over a
// map's outputs (32 rows apart in shared memory: bank conflicts) took 39.7 and
// 34.3 ms.
// ---------------------------------------------------------------------------
namespace fmm {

constexpr int ROT_MAXP = 16, ROT_ROWS = 32;
constexpr int ROT_LD = ROT_ROWS + 1;  // row pitch of [coefficient][target]: transposed writes without bank conflicts
constexpr int ROT_G = 40;  // factors per vector: g_l = l!/|u|^(l+1), l <= 2 p - 2, zeros after

// the jobs of every warp and where each map starts in a polar angle's table
struct RotPlan {
    int off[2][ROT_MAXP + 1];     // [part][K]: part 0 real (K = n + 1), 1 imaginary (K = n)
    int ds;                       // entries of one table
    unsigned char njob[8];
    unsigned char job[8][32];     // K | part << 7
    unsigned char nm[ROT_MAXP * (ROT_MAXP + 1) / 2][2];  // coefficient pair -> degree, order
};

// Entries per vector: the phases e^{ima} as the pairs that make the real part
// of a product, (cos, -sin), and the imaginary part, (sin, cos); then the
// factors from g_0, g_1, g_2 and g_3 on, so that a window of them starting
// anywhere is aligned in one of the copies.
constexpr int ROT_PH = 2 * ROT_MAXP, ROT_VS = 2 * ROT_PH + 4 * ROT_G;

// Inside the kernel the coefficients of a degree are in the order Re (n, 0) ..
// Re (n, n), Im (n, 1) .. Im (n, n): entry i of a (degree, part) job.
__host__ __device__ constexpr int rot_idx(int n, int part, int i) { return n * n + part * (n + 1) + i; }

template <class T>
struct RotVec;
template <>
struct RotVec<float> {
    using type = float4;
    static constexpr int n = 4;
};
template <>
struct RotVec<double> {
    using type = double2;
    static constexpr int n = 2;
};

// K rounded up to whole 16-byte vectors: the length of a map's rows
template <class T>
static int rot_pad(int K) { return (K + RotVec<T>::n - 1) / RotVec<T>::n * RotVec<T>::n; }

template <class T>
static RotPlan rot_plan(int p, int W)
{
    RotPlan P;
    std::memset(&P, 0, sizeof(P));
    std::vector<std::pair<int, int>> jobs;  // (K, part), largest first
    for (int part = 0; part < 2; part++)
        for (int K = 1; K <= p - part; K++) {
            P.off[part][K] = P.ds;
            P.ds += K * rot_pad<T>(K);
            jobs.push_back({K, part});
        }
    std::sort(jobs.begin(), jobs.end(), [](auto &x, auto &y) { return x.first != y.first ? x.first > y.first : x.second < y.second; });
    int load[8] = {};
    for (auto &j : jobs) {
        int w = 0;
        for (int k = 1; k < W; k++)
            if (load[k] < load[w]) w = k;
        load[w] += j.first * rot_pad<T>(j.first) + 8;
        P.job[w][P.njob[w]++] = (unsigned char)(j.first | j.second << 7);
    }
    int q = 0;
    for (int n = 0; n < p; n++)
        for (int m = 0; m <= n; m++, q++) {
            P.nm[q][0] = (unsigned char)n;
            P.nm[q][1] = (unsigned char)m;
        }
    return P;
}

// Host image, FP64: per distinct polar angle the maps (rows unpadded, parts and
// sizes in order), per vector its angle, phases and factors. One per process
// for each (p, MAC constant, stencil bound).
struct RotImage {
    int na = 0;
    std::vector<double> maps;   // na x sum K^2
    std::vector<int> angle;     // per vector
    std::vector<double> vec;    // per vector ROT_VS
};
static std::mutex g_rot_mu;
static std::map<std::tuple<int, double, int>, std::shared_ptr<const RotImage>> g_rot_cache;

// run f(0 .. count - 1) on the host cores; the first exception is rethrown
template <class F>
static void host_parallel(int count, F f)
{
    const unsigned nt = std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
    auto stride = [&](unsigned t) {
        for (int i = (int)t; i < count; i += (int)nt) f(i);
    };
    std::vector<std::thread> pool;
    std::vector<std::exception_ptr> fault(nt);  // an exception stays in its thread until the join
    unsigned started = 0;
    try {
        for (; started < nt; started++)
            pool.emplace_back([&, started] {
                try {
                    stride(started);
                } catch (...) {
                    fault[started] = std::current_exception();
                }
            });
    } catch (...) {
        // a thread could not be created: the strides without a thread run here
    }
    for (unsigned t = started; t < nt; t++) {
        try {
            stride(t);
        } catch (...) {
            fault[t] = std::current_exception();
            break;
        }
    }
    for (auto &th : pool) th.join();
    for (auto &e : fault)
        if (e) std::rethrow_exception(e);
}

static std::shared_ptr<const RotImage> rot_image(fmm_ctx *h)
{
    const auto key = std::make_tuple(h->p, h->cmac, h->st_R);
    {
        std::lock_guard<std::mutex> lk(g_rot_mu);
        auto it = g_rot_cache.find(key);
        if (it != g_rot_cache.end()) return it->second;
    }
    const int p = h->p, nv = h->nV;
    auto img = std::make_shared<RotImage>();
    img->angle.assign((size_t)nv, 0);
    img->vec.assign((size_t)nv * ROT_VS, 0.0);
    std::map<std::pair<int, int>, int> angles;  // (u_z, u_x^2 + u_y^2)
    std::vector<double> beta;
    const int ne = h->st_off[8];
    for (int e = 0; e < ne; e++) {
        const int *v = &h->st_host[4 * (size_t)e];
        const int id = v[3] & 0xffff;
        // u = c_L - c_M = -(source - target)
        const double u[3] = {-(double)v[0], -(double)v[1], -(double)v[2]};
        const double rxy = std::hypot(u[0], u[1]), a = rxy > 0 ? std::atan2(u[1], u[0]) : 0.0;
        auto it = angles.emplace(std::make_pair(-v[2], v[0] * v[0] + v[1] * v[1]), (int)beta.size());
        if (it.second) beta.push_back(std::atan2(rxy, u[2]));
        img->angle[(size_t)id] = it.first->second;
        double *o = img->vec.data() + (size_t)id * ROT_VS;
        for (int m = 0; m < p; m++) {
            const double co = std::cos(m * a), si = std::sin(m * a);
            o[2 * m] = co;
            o[2 * m + 1] = -si;
            o[ROT_PH + 2 * m] = si;
            o[ROT_PH + 2 * m + 1] = co;
        }
        const double d = std::sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        double g = 1.0 / d;
        for (int l = 0; l < 2 * p - 1; l++) {
            if (l) g *= (double)l / d;
            for (int k = 0; k <= std::min(l, 3); k++) o[2 * ROT_PH + k * ROT_G + l - k] = g;
        }
    }
    img->na = (int)beta.size();
    size_t per = 0;
    for (int K = 1; K <= p; K++) per += (size_t)K * K + (K < p ? (size_t)K * K : 0);
    img->maps.assign((size_t)img->na * per, 0.0);
    host_parallel(img->na, [&](int i) {
        const auto V = vmaps(p, beta[(size_t)i]);
        double *o = img->maps.data() + (size_t)i * per;
        for (int part = 0; part < 2; part++)
            for (int K = 1; K <= p - part; K++) {
                const int n = part ? K : K - 1, S = 2 * n + 1;
                for (int m = part; m <= n; m++)
                    for (int mp = part; mp <= n; mp++) {
                        const double s = ((m & 1) ? -1.0 : 1.0) * V[n][(size_t)(n - m) * S + n + mp];
                        const double t = V[n][(size_t)(n + m) * S + n + mp];
                        *o++ = (part ? t - s : t + s) / std::sqrt(fact(n + mp) * fact(n - mp));
                    }
            }
    });
    std::lock_guard<std::mutex> lk(g_rot_mu);
    g_rot_cache[key] = img;
    return img;
}

// device copy: maps (padded rows), vectors, c per coefficient pair and (halved
// for order 0) per coefficient, angle indices
template <class T>
static void rotation_tables_update(fmm_ctx *h, const RotPlan &P)
{
    const int want = sizeof(T) == 8 ? 2 : 1;
    if (h->rot_nv == h->nV && h->rot_kind == want && h->rot_tab.p) return;
    auto img = rot_image(h);
    const int p = h->p;
    std::vector<T> buf((size_t)img->na * P.ds + (size_t)h->nV * ROT_VS + ROT_MAXP * (ROT_MAXP + 1) / 2 + ROT_MAXP * ROT_MAXP, T(0));
    const double *in = img->maps.data();
    for (int i = 0; i < img->na; i++)
        for (int part = 0; part < 2; part++)
            for (int K = 1; K <= p - part; K++) {
                T *o = buf.data() + (size_t)i * P.ds + P.off[part][K];
                for (int r = 0; r < K; r++)
                    for (int c = 0; c < K; c++) o[r * rot_pad<T>(K) + c] = (T)*in++;
            }
    h->rot_vec_off = (size_t)img->na * P.ds;
    for (size_t i = 0; i < img->vec.size(); i++) buf[h->rot_vec_off + i] = (T)img->vec[i];
    h->rot_c_off = h->rot_vec_off + img->vec.size();
    for (int n = 0, q = 0; n < p; n++)
        for (int m = 0; m <= n; m++, q++) {
            const T c = (T)std::sqrt(fact(n + m) * fact(n - m));
            buf[h->rot_c_off + q] = c;
            T *ck = buf.data() + h->rot_c_off + ROT_MAXP * (ROT_MAXP + 1) / 2;
            ck[rot_idx(n, 0, m)] = m ? c : T(0.5) * c;
            if (m) ck[rot_idx(n, 1, m - 1)] = c;
        }
    h->rot_tab.ensure(sizeof(T) * buf.size());
    FMM_CUDA_TRY(cudaMemcpy(h->rot_tab.p, buf.data(), sizeof(T) * buf.size(), cudaMemcpyHostToDevice));
    h->rot_angle.ensure(sizeof(int) * img->angle.size());
    FMM_CUDA_TRY(cudaMemcpy(h->rot_angle.p, img->angle.data(), sizeof(int) * img->angle.size(), cudaMemcpyHostToDevice));
    h->rot_nv = h->nV;
    h->rot_kind = want;
}

// sum of one coefficient over the vectors: FP64, or an FP32 TwoSum pair
template <class T>
struct RotSum;
template <>
struct RotSum<double> {
    double s;
    __device__ __forceinline__ void zero() { s = 0.0; }
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double get() const { return s; }
    using part = double;
    __device__ __forceinline__ double pack() const { return s; }
    __device__ __forceinline__ void merge(double v) { s += v; }
};
template <>
struct RotSum<float> {
    float hi, lo;
    __device__ __forceinline__ void zero() { hi = lo = 0.f; }
    __device__ __forceinline__ void add(float v)
    {
        const float s = hi + v, b = s - hi;
        lo += (hi - (s - b)) + (v - b);
        hi = s;
    }
    __device__ __forceinline__ float get() const { return hi + lo; }
    using part = float2;
    __device__ __forceinline__ float2 pack() const { return make_float2(hi, lo); }
    __device__ __forceinline__ void merge(float2 v)
    {
        add(v.x);
        lo += v.y;
    }
};

// Runs of 16 bytes of T against scalars and runs: FP32 as packed pairs (one
// instruction for two multiply-adds, and half the issue slots).
template <class T>
struct RotPk;
template <>
struct RotPk<float> {
    using type = unsigned long long;
    static constexpr int n = 2;  // values per register pair
    static __device__ __forceinline__ type dup(float a)
    {
        type d;
        asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
        return d;
    }
    static __device__ __forceinline__ type make(float a, float b)
    {
        type d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
        return d;
    }
    static __device__ __forceinline__ void get(type v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
    static __device__ __forceinline__ void mad(type &acc, type a, type b)
    {
        asm("fma.rn.ftz.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
    }
};

// forward: outputs in registers, one input (with its phase) and one map row at
// a time; from the gathered rows r to x
template <class T, int NC>
__device__ __forceinline__ void rot_forward(const T *r, T *x, const T *ph, const T *map, int K, int n, int part)
{
    const T *re = r + (n * n + part) * ROT_LD, *im = r + rot_idx(n, 1, part - 1) * ROT_LD;
    // order 0 has no imaginary part: its sine is 0, and the value read in its
    // place is the degree's last real one
    const T *pp = ph + part * (ROT_PH + 2);
    T *out = x + rot_idx(n, part, 0) * ROT_LD;
    if constexpr (sizeof(T) == 4) {
        using P = RotPk<float>;
        unsigned long long o[2 * NC];
#pragma unroll
        for (int j = 0; j < 2 * NC; j++) o[j] = 0ull;
        const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(map);
#pragma unroll 2
        for (int i = 0; i < K; i++, row += NC, re += ROT_LD, im += ROT_LD, pp += 2) {
            const float2 w = *reinterpret_cast<const float2 *>(pp);
            const unsigned long long a = P::dup(*re * w.x + *im * w.y);
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const ulonglong2 d = row[c];
                P::mad(o[2 * c], d.x, a);
                P::mad(o[2 * c + 1], d.y, a);
            }
        }
#pragma unroll
        for (int c = 0; c < 2 * NC; c++) {
            float a, b;
            P::get(o[c], a, b);
            if (2 * c < 4 * NC - 3 || 2 * c < K) out[2 * c * ROT_LD] = a;
            if (2 * c + 1 < 4 * NC - 3 || 2 * c + 1 < K) out[(2 * c + 1) * ROT_LD] = b;
        }
    } else {
        T o[2 * NC];
#pragma unroll
        for (int j = 0; j < 2 * NC; j++) o[j] = T(0);
        const double2 *row = reinterpret_cast<const double2 *>(map);
#pragma unroll 2
        for (int i = 0; i < K; i++, row += NC, re += ROT_LD, im += ROT_LD, pp += 2) {
            const double2 w = *reinterpret_cast<const double2 *>(pp);
            const T a = *re * w.x + *im * w.y;
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const double2 d = row[c];
                o[2 * c] += d.x * a;
                if (c < NC - 1 || 2 * NC == K) o[2 * c + 1] += d.y * a;
            }
        }
#pragma unroll
        for (int j = 0; j < 2 * NC; j++)
            if (j < 2 * NC - 1 || j < K) out[j * ROT_LD] = o[j];
    }
}

// back: inputs in registers, one output at a time
template <class T, int NC>
__device__ __forceinline__ void rot_back(T *x, const T *map, int K, int n, int part)
{
    T *v = x + rot_idx(n, part, 0) * ROT_LD;
    if constexpr (sizeof(T) == 4) {
        using P = RotPk<float>;
        unsigned long long r[2 * NC];
#pragma unroll
        for (int c = 0; c < 2 * NC; c++)
            r[c] = P::make(2 * c < 4 * NC - 3 || 2 * c < K ? v[2 * c * ROT_LD] : 0.f,
                           2 * c + 1 < 4 * NC - 3 || 2 * c + 1 < K ? v[(2 * c + 1) * ROT_LD] : 0.f);
        const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(map);
#pragma unroll 2
        for (int i = 0; i < K; i++, row += NC, v += ROT_LD) {
            unsigned long long s0 = 0ull, s1 = 0ull;
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const ulonglong2 d = row[c];
                P::mad(s0, d.x, r[2 * c]);
                P::mad(s1, d.y, r[2 * c + 1]);
            }
            float a, b, c, d;
            P::get(s0, a, b);
            P::get(s1, c, d);
            *v = (a + b) + (c + d);
        }
    } else {
        T r[2 * NC];
#pragma unroll
        for (int j = 0; j < 2 * NC; j++) r[j] = j < 2 * NC - 1 || j < K ? v[j * ROT_LD] : T(0);
        const double2 *row = reinterpret_cast<const double2 *>(map);
#pragma unroll 2
        for (int i = 0; i < K; i++, row += NC, v += ROT_LD) {
            T s0 = 0, s1 = 0;
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const double2 d = row[c];
                s0 += d.x * r[2 * c];
                if (c < NC - 1 || 2 * NC == K) s1 += d.y * r[2 * c + 1];
            }
            *v = s0 + s1;
        }
    }
}

// along z: order m = p - K, out_n = +-sum_j g_{j+n} in_j over the degrees m .. p-1
// (order m of degree n is entry m - part of its part)
template <class T, int NC>
__device__ __forceinline__ void rot_along(T *x, const T *g, int K, int m, int part)
{
    constexpr int VN = RotVec<T>::n;
    // rot_idx(n, part, m - part): steps of 2 n + 1 + part from degree to degree
    T *const x0 = x + rot_idx(m, part, m - part) * ROT_LD;
    const int d0 = (2 * m + 1 + part) * ROT_LD;
    const T sg = (part ? T(-1) : T(1)) * (m == 0 ? T(0.5) : T(1));  // and alternating with the degree
    T r[NC * VN];
    {
        const T *v = x0;
        int d = d0;
#pragma unroll
        for (int j = 0; j < NC * VN; j++) {
            r[j] = j < (NC - 1) * VN + 1 || j < K ? *v : T(0);
            if (j + 1 < (NC - 1) * VN + 1 || j + 1 < K) v += d;
            d += 2 * ROT_LD;
        }
    }
    T *v = x0;
    int d = d0;
    if constexpr (sizeof(T) == 4) {
        using P = RotPk<float>;
        unsigned long long rp[2 * NC];
#pragma unroll
        for (int c = 0; c < 2 * NC; c++) rp[c] = P::make(r[2 * c], r[2 * c + 1]);
        // windows of factors for outputs nn .. nn + 3: from g_{2m + nn}, and from
        // the next one for the odd outputs
        const int sh = 2 * (m & 1);
        const ulonglong2 *wa = reinterpret_cast<const ulonglong2 *>(g + sh * ROT_G + 2 * m - sh);
        const ulonglong2 *wb = reinterpret_cast<const ulonglong2 *>(g + (sh + 1) * ROT_G + 2 * m - sh);
        for (int nn = 0; nn < K; nn += 4, wa++, wb++) {
            unsigned long long a[2 * NC + 2], b[2 * NC + 2];
#pragma unroll
            for (int c = 0; c <= NC; c++) {
                const ulonglong2 u = wa[c], w = wb[c];
                a[2 * c] = u.x;
                a[2 * c + 1] = u.y;
                b[2 * c] = w.x;
                b[2 * c + 1] = w.y;
            }
            unsigned long long s[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
            for (int c = 0; c < 2 * NC; c++) {
                P::mad(s[0], a[c], rp[c]);
                P::mad(s[1], b[c], rp[c]);
                P::mad(s[2], a[c + 1], rp[c]);
                P::mad(s[3], b[c + 1], rp[c]);
            }
#pragma unroll
            for (int o = 0; o < 4; o++) {
                float lo, hi;
                P::get(s[o], lo, hi);
                if (nn + o < K) *v = (lo + hi) * (o & 1 ? -sg : sg);
                v += d;
                d += 2 * ROT_LD;
            }
        }
    } else {
        const double2 *w = reinterpret_cast<const double2 *>(g + 2 * m);
        for (int nn = 0; nn < K; nn += 2, w++) {
            T gw[2 * NC + 2];
#pragma unroll
            for (int c = 0; c <= NC; c++) {
                const double2 u = w[c];
                gw[2 * c] = u.x;
                gw[2 * c + 1] = u.y;
            }
            T s[4] = {0, 0, 0, 0};
#pragma unroll
            for (int c = 0; c < NC; c++) {
                s[0] += gw[2 * c] * r[2 * c];
                s[1] += gw[2 * c + 1] * r[2 * c];
                if (c < NC - 1 || 2 * NC == K) {
                    s[2] += gw[2 * c + 1] * r[2 * c + 1];
                    s[3] += gw[2 * c + 2] * r[2 * c + 1];
                }
            }
#pragma unroll
            for (int o = 0; o < 2; o++) {
                if (nn + o < K) *v = (s[o] + s[o + 2]) * (o ? -sg : sg);
                v += d;
                d += 2 * ROT_LD;
            }
        }
    }
}

#define ROT_CASES(NCV, CALL)          \
    switch (NCV) {                    \
    case 1: CALL(1); break;           \
    case 2: CALL(2); break;           \
    case 3: CALL(3); break;           \
    case 4: CALL(4); break;           \
    default:                          \
        if constexpr (NCMAX > 4) {    \
            switch (NCV) {            \
            case 5: CALL(5); break;   \
            case 6: CALL(6); break;   \
            case 7: CALL(7); break;   \
            default: CALL(8); break;  \
            }                         \
        }                             \
    }

struct RotJob {
    const M2LTile *tiles;
    const int *ntiles, *tgt;
    const int4 *xyz;
    const uint64_t *anchor;
    const LevelDesc *ld;
    const int *map_pool;
    const int4 *st;
    const int *st_off;
    const int *angle;
    unsigned *tcnt;
    void *part;
    int nsplit, chunk;
};

// c M~ of the cells from level 2 on (halved for order 0, as the forward maps
// take it), in the kernel's coefficient order
template <class T>
__global__ void __launch_bounds__(256) rot_scale_k(const T *__restrict__ M, int PP, int c0, int nc, const T *__restrict__ ck,
                                                   T *__restrict__ CM)
{
    const int64_t i = (int64_t)c0 * PP + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nc * PP) return;
    const int k = (int)(i % PP);
    int n = 0;
    while ((n + 1) * (n + 1) <= k) n++;
    const int j = k - n * n;  // Re 0, then Re and Im of 1 .. n
    const int o = rot_idx(n, j && !(j & 1), j & 1 ? (j + 1) / 2 : j ? j / 2 - 1 : 0);
    CM[i - k + o] = M[i] * ck[o];
}

// Lookups on levels without a dense map, kept out of the kernel's registers: N
// = 60,001, p = 16 takes 7.9 ms, with them in line 8.5.
static __device__ __noinline__ int rot_lookup(const LevelDesc *L, const int *map_pool, const uint64_t *anchor, int l, int x, int y,
                                              int z)
{
    return level_lookup(*L, map_pool, anchor, l, x, y, z);
}

// W warps, NQ >= p (p + 1) / 2 / W coefficient pairs per warp
template <class T, int W, int NQ>
__global__ void __launch_bounds__(32 * W, W == 8 ? 2 : NQ > 9 ? 3 : 4)
    m2l_rot_k(int p, const __grid_constant__ RotJob J, const __grid_constant__ RotPlan P, const T *__restrict__ maps,
              const T *__restrict__ vecs, const T *__restrict__ cfac, const T *__restrict__ CM, T *__restrict__ L)
{
    using S = RotSum<T>;
    using V = typename RotVec<T>::type;
    constexpr int VN = RotVec<T>::n, NCMAX = ROT_MAXP / VN;
    if ((int)blockIdx.x >= *J.ntiles * J.nsplit) return;
    const int tile = (int)blockIdx.x / J.nsplit, split = (int)blockIdx.x - tile * J.nsplit;
    const M2LTile td = J.tiles[tile];
    const int PP = p * p, npair = p * (p + 1) / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // two buffers of a vector's phases and factors and its maps, then the
    // gathered rows and the coefficients in work
    T *const sv = reinterpret_cast<T *>(smem_raw);
    const int vstep = ROT_VS + P.ds;
    T *const sr = sv + 2 * vstep, *const sx = sr + (size_t)PP * ROT_LD;
    __shared__ int s_last;
    __shared__ int4 s_pair[W * NQ];  // coefficient pair -> rows of its parts, 2 m
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T *x = sx + lane;
    int cell = -1, rl = td.level, px = 0, py = 0, pz = 0, ro = 0;
    if (lane < td.count) {
        cell = J.tgt[td.start + lane];
        const int4 a = J.xyz[cell];
        rl = a.w;
        const int sh = FMM_MAXLEVEL - rl;
        px = a.x >> sh;
        py = a.y >> sh;
        pz = a.z >> sh;
        ro = (px & 1) | ((py & 1) << 1) | ((pz & 1) << 2);
    }
    for (int q = threadIdx.x; q < npair; q += 32 * W) {
        const int n = P.nm[q][0], m = P.nm[q][1];
        s_pair[q] = make_int4(rot_idx(n, 0, m) * ROT_LD, rot_idx(n, m ? 1 : 0, m ? m - 1 : 0) * ROT_LD, 2 * m, 0);
    }
    // source lookups: the first cell of a level with every lattice cell, the
    // level's dense map, or neither (-1)
    const LevelDesc *ld = J.ld + rl;
    const bool whole = rl <= 10 && ld->end - ld->start == (1 << (3 * rl));
    const int start = ld->start;
    const int *const map = ld->map_off >= 0 && ld->up == 0 ? J.map_pool + ld->map_off : nullptr;
    S acc[2 * NQ];
#pragma unroll
    for (int k = 0; k < 2 * NQ; k++) acc[k].zero();
    // the set's entries are sorted by reach: only a prefix can hit a cell;
    // this CTA's range of it
    const int nvt = J.st_off[10 + td.octant * (FMM_MAXLEVEL + 1) + td.level];
    // (ranges of a fixed length: a cell's sums do not depend on its tile's list)
    int e = J.st_off[td.octant] + min(nvt, split * J.chunk);
    const int e1 = J.st_off[td.octant] + (split + 1 < J.nsplit ? min(nvt, (split + 1) * J.chunk) : nvt);

    // next entry from e on that hits a cell of some lane (every warp finds the
    // same), with this lane's source cell
    auto advance = [&](int &id, int &src) {
        for (; e < e1; e++) {
            const int4 v = J.st[e];
            int b = -1;
            if (cell >= 0 && ((v.w >> (16 + ro)) & 1)) {
                const int qx = px + v.x, qy = py + v.y, qz = pz + v.z;
                const unsigned side = 1u << rl;
                if ((unsigned)qx < side && (unsigned)qy < side && (unsigned)qz < side)
                    b = whole ? start + (int)morton3_10((uint32_t)qx, (uint32_t)qy, (uint32_t)qz)
                        : map ? map[morton3_10((uint32_t)qx, (uint32_t)qy, (uint32_t)qz)]
                              : rot_lookup(ld, J.map_pool, J.anchor, rl, qx, qy, qz);
            }
            if (__any_sync(0xffffffffu, b >= 0)) {
                id = v.w & 0xffff;
                src = b;
                e++;
                return true;
            }
        }
        return false;
    };
    auto fetch = [&](int id, int buf) {
        const V *gv = reinterpret_cast<const V *>(vecs + (size_t)id * ROT_VS);
        const V *gm = reinterpret_cast<const V *>(maps + (size_t)J.angle[id] * P.ds);
        for (int i = threadIdx.x; i < ROT_VS / VN; i += 32 * W) cp_async16(smem_u32(sv + buf * vstep + i * VN), gv + i, 16);
        for (int i = threadIdx.x; i < P.ds / VN; i += 32 * W) cp_async16(smem_u32(sv + buf * vstep + ROT_VS + i * VN), gm + i, 16);
    };
    auto gather = [&](int src) {
#pragma unroll 2
        for (int r = warp; r < ROT_ROWS; r += W) {
            const int b = __shfl_sync(0xffffffffu, src, r);
            const T *row = CM + (size_t)(b >= 0 ? b : 0) * PP;
            for (int j = lane; j < PP; j += 32) cp_async_n<sizeof(T)>(smem_u32(sr + j * ROT_LD + r), row + j, b >= 0);
        }
    };

    int id = 0, src = -1, buf = 0;
    bool have = advance(id, src);
    if (have) {
        fetch(id, 0);
        gather(src);
    }
    while (have) {
        have = advance(id, src);
        cp_async_wait_all();
        __syncthreads();  // the vector's data is here, and no warp reads the other buffer any more
        const T *ph = sv + buf * vstep, *g = ph + 2 * ROT_PH, *mp = ph + ROT_VS;
        for (int j = 0; j < P.njob[warp]; j++) {
            const int K = P.job[warp][j] & 127, part = P.job[warp][j] >> 7, n = part ? K : K - 1;
#define ROT_CALL(NC) rot_forward<T, NC>(sr + lane, x, ph, mp + P.off[part][K], K, n, part)
            ROT_CASES((K + VN - 1) / VN, ROT_CALL)
#undef ROT_CALL
        }
        __syncthreads();
        if (have) {  // the gathered rows are used up
            fetch(id, buf ^ 1);
            gather(src);
        }
        for (int j = 0; j < P.njob[warp]; j++) {
            const int K = P.job[warp][j] & 127, part = P.job[warp][j] >> 7;
#define ROT_CALL(NC) rot_along<T, NC>(x, g, K, p - K, part)
            ROT_CASES((K + VN - 1) / VN, ROT_CALL)
#undef ROT_CALL
        }
        __syncthreads();
        for (int j = 0; j < P.njob[warp]; j++) {
            const int K = P.job[warp][j] & 127, part = P.job[warp][j] >> 7, n = part ? K : K - 1;
#define ROT_CALL(NC) rot_back<T, NC>(x, mp + P.off[part][K], K, n, part)
            ROT_CASES((K + VN - 1) / VN, ROT_CALL)
#undef ROT_CALL
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NQ; k++) {
            const int q = min(warp + W * k, npair - 1);  // (a clamped pair's sums are not used)
            const int4 s = s_pair[q];
            const T yr = x[s.x], yi = x[s.y], si = ph[ROT_PH + s.z], co = ph[ROT_PH + s.z + 1];
            acc[2 * k].add(yr * co - yi * si);
            acc[2 * k + 1].add(yr * si + yi * co);  // m = 0: not used
        }
        buf ^= 1;
    }
    auto put = [&](int q, const S &re, const S &im) {
        if (cell < 0) return;
        const int n = P.nm[q][0], m = P.nm[q][1];
        T *Lc = L + (size_t)cell * PP;
        Lc[re_idx(n, m)] += re.get() * cfac[q];
        if (m) Lc[im_idx(n, m)] += im.get() * cfac[q];
    };
    if (J.nsplit == 1) {
#pragma unroll
        for (int k = 0; k < NQ; k++)
            if (warp + W * k < npair) put(warp + W * k, acc[2 * k], acc[2 * k + 1]);
        return;
    }
    // the range's sums, [item][pair][re, im][lane]; the tile's last range to
    // finish adds them all in order
    using Pt = typename S::part;
    Pt *part = static_cast<Pt *>(J.part);
    const size_t rng = (size_t)npair * 2 * ROT_ROWS;
    Pt *mine = part + (size_t)blockIdx.x * rng + lane;
#pragma unroll
    for (int k = 0; k < NQ; k++) {
        const int q = warp + W * k;
        if (q >= npair) break;
        __stcg(&mine[(size_t)(2 * q) * ROT_ROWS], acc[2 * k].pack());
        __stcg(&mine[(size_t)(2 * q + 1) * ROT_ROWS], acc[2 * k + 1].pack());
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(&J.tcnt[tile], 1u) == (unsigned)(J.nsplit - 1);
        if (s_last) J.tcnt[tile] = 0u;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    const Pt *first = part + (size_t)tile * J.nsplit * rng + lane;
    for (int q = warp; q < npair; q += W) {
        S re, im;
        re.zero();
        im.zero();
#pragma unroll 4
        for (int r = 0; r < J.nsplit; r++) {
            re.merge(__ldcg(&first[(size_t)r * rng + (size_t)(2 * q) * ROT_ROWS]));
            im.merge(__ldcg(&first[(size_t)r * rng + (size_t)(2 * q + 1) * ROT_ROWS]));
        }
        put(q, re, im);
    }
}

// Ranges per tile: about 8 CTAs per SM, so that the tiles at the boundary of
// the domain, which have fewer sources, even out, of 24 vectors or more. Part of
// the build, which fixes the tiles (the pooling threshold may be set anew before
// the next evaluation): the ranges cover the longest list of these tiles.
void rotation_plan(fmm_ctx *h)
{
    if (h->engine_used != FMM_M2L_ROTATION) return;
    const int nv = m2l_longest_list(h);
    const int fill = (8 * h->nsm + h->ntiles_max - 1) / std::max(h->ntiles_max, 1);
    const int want = std::max(1, std::min(fill, std::min(nv / 24, 32)));
    h->m2l_chunk = (nv + want - 1) / want;
    h->m2l_nsplit = (nv + h->m2l_chunk - 1) / h->m2l_chunk;
}

template <class T, int W, int NQ>
static void launch_rot(fmm_ctx *h, T *L, const T *M)
{
    const int p = h->p;
    const RotPlan P = rot_plan<T>(p, W);
    rotation_tables_update<T>(h, P);
    RotJob j;
    j.chunk = h->m2l_chunk;
    j.nsplit = h->m2l_nsplit;
    h->m2l_ws.ensure(sizeof(unsigned) * (size_t)h->ntiles_max);
    if (j.nsplit > 1) h->m2l_part.ensure(sizeof(double) * (size_t)h->ntiles_max * j.nsplit * p * (p + 1) * ROT_ROWS);
    FMM_CUDA_TRY(cudaMemsetAsync(h->m2l_ws.p, 0, sizeof(unsigned) * (size_t)h->ntiles_max, h->work));
    j.tiles = h->m2l_tiles.as<M2LTile>();
    j.ntiles = reinterpret_cast<const int *>(h->m2l_misc.as<unsigned>() + 24 * (FMM_MAXLEVEL + 1));
    j.tgt = h->m2l_tgt.as<int>();
    j.xyz = h->c_xyz.as<int4>();
    j.anchor = h->c_anchor.as<uint64_t>();
    j.ld = h->lvl_desc.as<LevelDesc>();
    j.map_pool = h->map_pool.as<int>();
    j.st = h->st_dev.as<int4>();
    j.st_off = stencil_offsets(h);
    j.angle = h->rot_angle.as<int>();
    j.tcnt = h->m2l_ws.as<unsigned>();
    j.part = h->m2l_part.p;
    const size_t smem = sizeof(T) * (2 * (size_t)p * p * ROT_LD + 2 * ((size_t)ROT_VS + P.ds));
    ensure_smem((const void *)m2l_rot_k<T, W, NQ>, smem);
    const T *tab = h->rot_tab.as<T>();
    const int c0 = h->lvl_start[2], nc = h->ncells, PP = p * p;
    h->rot_m.ensure(sizeof(T) * (size_t)nc * PP);
    if (nc <= c0) return;
    rot_scale_k<T><<<(unsigned)(((int64_t)(nc - c0) * PP + 255) / 256), 256, 0, h->work>>>(
        M, PP, c0, nc, tab + h->rot_c_off + ROT_MAXP * (ROT_MAXP + 1) / 2, h->rot_m.as<T>());
    count_launch(h);
    m2l_rot_k<T, W, NQ><<<(unsigned)h->ntiles_max * j.nsplit, 32 * W, smem, h->work>>>(
        p, j, P, tab, tab + h->rot_vec_off, tab + h->rot_c_off, h->rot_m.as<T>(), L);
    count_launch(h);
    check_launch("m2l rotation");
}

// Eight warps share the 136 coefficient pairs of p = 16; up to p = 10 four do
// (the largest of the jobs is then no more than a warp's share of them).
template <class T>
void m2l_rotation(fmm_ctx *h, T *L, const T *M)
{
    if (h->p <= 8) launch_rot<T, 4, 9>(h, L, M);
    else if (h->p <= 10) launch_rot<T, 4, 14>(h, L, M);
    else launch_rot<T, 8, 17>(h, L, M);
}

template void m2l_rotation<float>(fmm_ctx *, float *, const float *);
template void m2l_rotation<double>(fmm_ctx *, double *, const double *);

bool rotation_m2l_supported(fmm_ctx *h) { return h->p >= 1 && h->p <= ROT_MAXP; }
int rotation_tile_rows(fmm_ctx *) { return ROT_ROWS; }

}  // namespace fmm
