// L-BFGS (Sec. 5.2) on the device in float64: deterministic dot products and
// the two-loop recursion with every scalar kept on the device, so a direction
// costs no host round trip. Vectors are the half-array modes viewed as 2*NH
// reals (real and imaginary parts are independent variables, Sec. 5.1).
//
// The recursion alternates a dot product with an update that needs its value.
// Each step is one pass over the vectors: it adds up the previous step's block
// partials (the same fixed order in every block), applies the update and forms
// the partials of the next dot product with the values it has just written. A
// step reads q, one history vector for the update and one for the dot, and
// writes q: 32 bytes an element, bound by memory. (As separate dot, reduction
// and update launches it was 40 bytes an element and three launches a step; a
// direction with 10 pairs at 192^3 took 1.85 ms.)
#include <type_traits>

#include "common.cuh"

namespace pmr {
namespace {

constexpr int kT = 256;
constexpr int kG = kLbfgsBlocks;  // a fixed grid, so that sums have a fixed order

// the block's sum of v, in every thread
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    __syncthreads();  // sh free
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kT / 32; ++w) t += sh[w];
    return t;
}

// sum of the kG block partials of an earlier launch, in every thread
__device__ __forceinline__ double part_sum(const double* __restrict__ part, double* sh) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < (kG + kT - 1) / kT; ++i) {
        const int j = i * kT + threadIdx.x;
        if (j < kG) v += part[j];
    }
    return block_sum(v, sh);
}

// W consecutive values: 2 where every vector of a launch starts on a 16-byte
// boundary and n is even, else 1
template <int W>
struct Val {
    double v[W];
};
template <int W>
__device__ __forceinline__ Val<W> ld(const double* p, int64_t i) {
    if constexpr (W == 2) {
        const double2 t = reinterpret_cast<const double2*>(p)[i];
        return {t.x, t.y};
    } else {
        return {p[i]};
    }
}
template <int W>
__device__ __forceinline__ void st(double* p, int64_t i, const Val<W>& v) {
    if constexpr (W == 2) reinterpret_cast<double2*>(p)[i] = make_double2(v.v[0], v.v[1]);
    else p[i] = v.v[0];
}

// use(index, load(index)) over the launch's share of n / W values, U at a time with all
// their loads issued first. REV: from the end. The steps of the recursion alternate, so
// that each begins with the part of q its predecessor wrote last, still in L2.
template <int W, int U, bool REV = false, class L, class F>
__device__ __forceinline__ void sweep(int64_t n, L load, F use) {
    const int64_t m = n / W, step = (int64_t)gridDim.x * kT;
    int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x;
    auto at = [&](int64_t j) { return REV ? m - 1 - j : j; };
    for (; i + (U - 1) * step < m; i += U * step) {
        decltype(load(i)) t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = load(at(i + u * step));
#pragma unroll
        for (int u = 0; u < U; ++u) use(at(i + u * step), t[u]);
    }
    for (; i < m; i += step) use(at(i), load(at(i)));
}

// The Gaussian prior's inverse Hessian D = P~(k) / w_k, diagonal over the half
// array, 0 at k = 0: the index arithmetic and the table.
struct Prior {
    FastDiv fP, fN;
    const double* inv_pow;
    int N;
    // D of mode i (entry i of the half array)
    __device__ __forceinline__ bool at(uint32_t i, double* wip) const {
        const uint32_t t = fP.div(i);
        const int kz = (int)(i - t * fP.d);
        const uint32_t ixu = fN.div(t);
        const int iy = (int)(t - ixu * fN.d), ix = (int)ixu;
        const int nx = 2 * ix <= N ? ix : ix - N, ny = 2 * iy <= N ? iy : iy - N;
        const double ip = inv_pow[nx * nx + ny * ny + kz * kz];
        *wip = ((kz == 0 || 2 * kz == N) ? 1.0 : 2.0) * ip;
        return ip > 0.0;
    }
};
// scale D x of the W values at i
template <int W>
__device__ __forceinline__ Val<W> prior_h0(const Prior& p, int64_t i, const Val<W>& x, double scale) {
    double wip;
    const bool nz = p.at((uint32_t)(i * W >> 1), &wip);
    Val<W> y;
#pragma unroll
    for (int k = 0; k < W; ++k) y.v[k] = nz ? scale * x.v[k] / wip : 0.0;
    return y;
}

template <int W>
struct Two {
    Val<W> a, b;
};
template <int W>
struct Three {
    Val<W> a, b, c;
};

// q = g, partials of w . q
template <int W>
__global__ void __launch_bounds__(kT, 4) k_copy_dot(double* __restrict__ q, const double* __restrict__ g,
                                                 const double* __restrict__ w, int64_t n, double* __restrict__ part) {
    __shared__ double sh[kT / 32];
    double acc = 0.0;
    sweep<W, 2>(n, [&](int64_t i) { return Two<W>{ld<W>(g, i), ld<W>(w, i)}; },
                [&](int64_t i, const Two<W>& t) {
                    st<W>(q, i, t.a);
#pragma unroll
                    for (int k = 0; k < W; ++k) acc = fma(t.b.v[k], t.a.v[k], acc);
                });
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// One step of the recursion; dot = the sum of part_in.
//  FIRST: alpha = rho dot;          q -= alpha x        (first loop, x = y_t)
//  SCALE: the same, then q = gamma H0 q, gamma = gs[0] / gs[1]  (its last step)
//  SECOND: beta = rho dot;          q += (alpha - beta) x  (second loop, x = s_t)
//  LAST: the same, then q = -q                          (its last step)
// then the partials of w . q. rho = 1 / *sy where sy is set.
enum Kind : int { FIRST = 0, SCALE = 1, SECOND = 2, LAST = 3 };
template <int W, int KIND, bool REV>
__global__ void __launch_bounds__(kT, 4) k_step(double* __restrict__ q, const double* x, const double* w, int64_t n,
                                             const double* __restrict__ part_in, double* __restrict__ part_out,
                                             double rho, const double* __restrict__ sy, double* __restrict__ alpha,
                                             const double* __restrict__ gs, bool use_prior, Prior pr) {
    __shared__ double sh[kT / 32];
    const double dot = part_sum(part_in, sh);
    if (sy) rho = 1.0 / *sy;
    double coef;
    if (KIND == FIRST || KIND == SCALE) {
        coef = -rho * dot;
        if (blockIdx.x == 0 && threadIdx.x == 0) *alpha = rho * dot;
    } else {
        coef = *alpha - rho * dot;
    }
    const double gamma = KIND == SCALE ? gs[0] / gs[1] : 1.0;
    double acc = 0.0;
    sweep<W, 2, REV>(n, [&](int64_t i) { return Three<W>{ld<W>(q, i), ld<W>(x, i), ld<W>(w, i)}; },
                [&](int64_t i, const Three<W>& t) {
                    Val<W> r;
#pragma unroll
                    for (int k = 0; k < W; ++k) r.v[k] = fma(coef, t.b.v[k], t.a.v[k]);
                    if (KIND == SCALE) {
                        if (use_prior) r = prior_h0<W>(pr, i, r, 1.0);
#pragma unroll
                        for (int k = 0; k < W; ++k) r.v[k] *= gamma;
                    }
                    if (KIND == LAST)
#pragma unroll
                        for (int k = 0; k < W; ++k) r.v[k] = -r.v[k];
                    st<W>(q, i, r);
#pragma unroll
                    for (int k = 0; k < W; ++k) acc = fma(t.c.v[k], r.v[k], acc);
                });
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part_out[blockIdx.x] = acc;
}

// Partials of s_t . y_t of pair t = blockIdx.y (vectors n apart) and, for the newest
// pair (the last), of y . H0 y: part[t][kG], then part[gridDim.y][kG].
template <int W>
__global__ void __launch_bounds__(kT, 4) k_pair_dots(const double* __restrict__ S, const double* __restrict__ Y, int64_t n,
                                                  bool use_prior, Prior pr, double* __restrict__ part) {
    __shared__ double sh[kT / 32];
    const double *s = S + blockIdx.y * n, *y = Y + blockIdx.y * n;
    const bool newest = blockIdx.y == gridDim.y - 1;
    double sy = 0.0, yy = 0.0;
    sweep<W, 2>(n, [&](int64_t i) { return Two<W>{ld<W>(s, i), ld<W>(y, i)}; },
                [&](int64_t i, const Two<W>& t) {
                    const Val<W> d = newest && use_prior ? prior_h0<W>(pr, i, t.b, 1.0) : t.b;
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        sy = fma(t.a.v[k], t.b.v[k], sy);
                        yy = fma(t.b.v[k], d.v[k], yy);
                    }
                });
    sy = block_sum(sy, sh);
    if (threadIdx.x == 0) part[blockIdx.y * kG + blockIdx.x] = sy;
    if (!newest) return;
    yy = block_sum(yy, sh);
    if (threadIdx.x == 0) part[gridDim.y * kG + blockIdx.x] = yy;
}

// out[b] = sum of part[b][kG], one block each
__global__ void __launch_bounds__(kT) k_part_sums(const double* __restrict__ part, double* __restrict__ out) {
    __shared__ double sh[kT / 32];
    const double t = part_sum(part + (int64_t)blockIdx.x * kG, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = t;
}

// y = scale D x and the partials of x . y
__global__ void __launch_bounds__(kT, 4) k_prior_h0_dot(double* __restrict__ y, const double* __restrict__ x, int64_t n,
                                                     Prior pr, double scale, double* __restrict__ part) {
    __shared__ double sh[kT / 32];
    double acc = 0.0;
    sweep<2, 4>(n, [&](int64_t i) { return ld<2>(x, i); },
                [&](int64_t i, const Val<2>& t) {
                    const Val<2> r = prior_h0<2>(pr, i, t, scale);
                    st<2>(y, i, r);
#pragma unroll
                    for (int k = 0; k < 2; ++k) acc = fma(t.v[k], r.v[k], acc);
                });
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// xt = x + t d, and s_k = xt in float32
__global__ void __launch_bounds__(kT) k_trial(double2* __restrict__ xt, const double2* __restrict__ x,
                                              const double2* __restrict__ d, double t, int64_t nh,
                                              float2* __restrict__ s_k) {
    const int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x;
    if (i >= nh) return;
    const double2 a = x[i], b = d[i];
    const double2 r = make_double2(fma(t, b.x, a.x), fma(t, b.y, a.y));
    xt[i] = r;
    s_k[i] = make_float2((float)r.x, (float)r.y);
}

__global__ void __launch_bounds__(kT) k_f64_to_c64(const double2* __restrict__ a, float2* __restrict__ out, int64_t nh) {
    const int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x;
    if (i < nh) out[i] = make_float2((float)a[i].x, (float)a[i].y);
}

// x and g from their float32 forms
__global__ void __launch_bounds__(kT) k_start(const float2* __restrict__ s_k, const float2* __restrict__ gk, int64_t nh,
                                              double2* __restrict__ x, double2* __restrict__ g) {
    const int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x;
    if (i >= nh) return;
    const float2 a = s_k[i], b = gk[i];
    x[i] = make_double2(a.x, a.y);
    g[i] = make_double2(b.x, b.y);
}

// The accepted point's gradient in float64, the candidate pair s = xt - x, y = gt - g,
// and the partials of s . y, s . s and y . y (part[3][kG]).
__global__ void __launch_bounds__(kT, 4) k_candidate(const float2* __restrict__ gk, const double* __restrict__ x,
                                                  const double* __restrict__ xt, const double* __restrict__ g,
                                                  int64_t n, double* __restrict__ gt, double* __restrict__ s,
                                                  double* __restrict__ y, double* __restrict__ part) {
    __shared__ double sh[kT / 32];
    struct In {
        Val<2> x, xt, g;
        float2 gk;
    };
    double sy = 0.0, ss = 0.0, yy = 0.0;
    sweep<2, 2>(n, [&](int64_t i) { return In{ld<2>(x, i), ld<2>(xt, i), ld<2>(g, i), gk[i]}; },
                [&](int64_t i, const In& t) {
                    const Val<2> gn{(double)t.gk.x, (double)t.gk.y};
                    Val<2> a, b;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        a.v[k] = t.xt.v[k] - t.x.v[k];
                        b.v[k] = gn.v[k] - t.g.v[k];
                        sy = fma(a.v[k], b.v[k], sy);
                        ss = fma(a.v[k], a.v[k], ss);
                        yy = fma(b.v[k], b.v[k], yy);
                    }
                    st<2>(gt, i, gn);
                    st<2>(s, i, a);
                    st<2>(y, i, b);
                });
    sy = block_sum(sy, sh);
    ss = block_sum(ss, sh);
    yy = block_sum(yy, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = sy;
        part[kG + blockIdx.x] = ss;
        part[2 * kG + blockIdx.x] = yy;
    }
}

Prior prior_of(const pmr_ctx* c) {
    return Prior{FastDiv((uint32_t)c->P), FastDiv((uint32_t)c->N), c->inv_power_tab, c->N};
}

template <int W>
int two_loop(pmr_ctx* c, const double* g, const double* S, const double* Y, int k, int head, int m, int64_t n,
             const double* rho_host, double* d, bool prior_h0) {
    pmr::LBFGS& L = c->lb;
    const Prior pr = prior_of(c);
    auto slot = [&](int t) { return (head + t) % m; };
    auto at = [&](const double* V, int t) { return V + (int64_t)slot(t) * n; };
    double* sums = L.sums;  // s.y of the k pairs (rho_host unset) or of the newest, then y.H0 y of the newest
    const int pairs = rho_host ? 1 : k;
    const double *S0 = rho_host ? at(S, k - 1) : S, *Y0 = rho_host ? at(Y, k - 1) : Y;
    k_pair_dots<W><<<dim3(kG, pairs), kT, 0, c->stream>>>(S0, Y0, n, prior_h0, pr, L.part + 2 * kG);
    PMR_TRY(check_launch(c, "pair_dots"));
    k_part_sums<<<pairs + 1, kT, 0, c->stream>>>(L.part + 2 * kG, sums);
    PMR_TRY(check_launch(c, "part_sums"));
    k_copy_dot<W><<<kG, kT, 0, c->stream>>>(d, g, at(S, k - 1), n, L.part);
    PMR_TRY(check_launch(c, "copy_dot"));
    int p = 0;
    // one step: dot partials at p, the next at p ^ 1, sweeping the other way round each time
    auto step = [&](auto kind, int t, const double* x, const double* w, const char* name) {
        constexpr int K = decltype(kind)::value;
        double *pin = L.part + p * kG, *pout = L.part + (p ^ 1) * kG, *al = L.alpha + slot(t);
        const double rho = rho_host ? rho_host[slot(t)] : 0.0;
        const double* sy = rho_host ? nullptr : sums + t;
        if (p)
            k_step<W, K, false><<<kG, kT, 0, c->stream>>>(d, x, w, n, pin, pout, rho, sy, al, sums + pairs - 1, prior_h0,
                                                          pr);
        else
            k_step<W, K, true><<<kG, kT, 0, c->stream>>>(d, x, w, n, pin, pout, rho, sy, al, sums + pairs - 1, prior_h0,
                                                         pr);
        p ^= 1;
        return check_launch(c, name);
    };
    using std::integral_constant;
    for (int t = k - 1; t > 0; --t)
        PMR_TRY(step(integral_constant<int, FIRST>{}, t, at(Y, t), at(S, t - 1), "two_loop_0"));
    PMR_TRY(step(integral_constant<int, SCALE>{}, 0, at(Y, 0), at(Y, 0), "two_loop_0"));
    for (int t = 0; t < k - 1; ++t)
        PMR_TRY(step(integral_constant<int, SECOND>{}, t, at(S, t), at(Y, t + 1), "two_loop_1"));
    PMR_TRY(step(integral_constant<int, LAST>{}, k - 1, at(S, k - 1), g, "two_loop_1"));
    k_part_sums<<<1, kT, 0, c->stream>>>(L.part + p * kG, L.scal);
    return check_launch(c, "part_sums");
}

}  // namespace

// d = -H g and scal[0] = g . d. S, Y are rings of capacity m: pair t (0 = oldest) sits in
// slot (head + t) % m. rho_host[slot] = 1 / (s.y) of that slot; NULL: formed here
// (head 0, m = k).
int lbfgs_two_loop(pmr_ctx* c, const double* g, const double* S, const double* Y, int k, int head, int m, int64_t n,
                   const double* rho_host, double* d, bool prior_h0) {
    const bool wide =
        n % 2 == 0 && (((uintptr_t)g | (uintptr_t)S | (uintptr_t)Y | (uintptr_t)d) & 15) == 0;
    return wide ? two_loop<2>(c, g, S, Y, k, head, m, n, rho_host, d, prior_h0)
                : two_loop<1>(c, g, S, Y, k, head, m, n, rho_host, d, prior_h0);
}

// d = -D g (the first direction of a stage) and scal[0] = g . d
int lbfgs_first_direction(pmr_ctx* c) {
    pmr::LBFGS& L = c->lb;
    k_prior_h0_dot<<<kG, kT, 0, c->stream>>>(L.d, L.g, L.n, prior_of(c), -1.0, L.part);
    PMR_TRY(check_launch(c, "prior_h0"));
    k_part_sums<<<1, kT, 0, c->stream>>>(L.part, L.scal);
    return check_launch(c, "part_sums");
}

int lbfgs_trial(pmr_ctx* c, double t, float2* s_k) {
    pmr::LBFGS& L = c->lb;
    k_trial<<<nblocks(c->NH, kT), kT, 0, c->stream>>>(reinterpret_cast<double2*>(L.xt),
                                                      reinterpret_cast<const double2*>(L.x),
                                                      reinterpret_cast<const double2*>(L.d), t, c->NH, s_k);
    return check_launch(c, "trial");
}

int lbfgs_start(pmr_ctx* c, const float2* s_k) {
    pmr::LBFGS& L = c->lb;
    k_start<<<nblocks(c->NH, kT), kT, 0, c->stream>>>(s_k, L.gk, c->NH, reinterpret_cast<double2*>(L.x),
                                                      reinterpret_cast<double2*>(L.g));
    return check_launch(c, "lbfgs_start");
}

int lbfgs_restore(pmr_ctx* c, float2* s_k) {
    k_f64_to_c64<<<nblocks(c->NH, kT), kT, 0, c->stream>>>(reinterpret_cast<const double2*>(c->lb.x), s_k, c->NH);
    return check_launch(c, "f64_to_c64");
}

// gt from gk, s into d, y into yk, and scal[0..2] = s.y, s.s, y.y
int lbfgs_candidate(pmr_ctx* c) {
    pmr::LBFGS& L = c->lb;
    k_candidate<<<kG, kT, 0, c->stream>>>(L.gk, L.x, L.xt, L.g, L.n, L.gt, L.d, L.yk, L.part);
    PMR_TRY(check_launch(c, "candidate"));
    k_part_sums<<<3, kT, 0, c->stream>>>(L.part, L.scal);
    return check_launch(c, "part_sums");
}

int lbfgs_alloc(pmr_ctx* c) {
    pmr::LBFGS& L = c->lb;
    L.m = c->cfg.lbfgs_m;
    L.n = 2 * c->NH;
    const size_t v = sizeof(double) * (size_t)L.n;
    PMR_TRY(check_cuda(c, cudaMalloc(&L.x, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.g, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.d, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.xt, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.gt, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.yk, v), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.S, v * L.m), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.Y, v * L.m), "lbfgs"));
    PMR_TRY(check_cuda(c, cudaMalloc(&L.alpha, sizeof(double) * lbfgs_scalars(L.m)), "lbfgs"));
    L.scal = L.alpha + L.m;
    L.sums = L.scal + 8;
    L.part = L.sums + L.m + 1;
    PMR_TRY(check_cuda(c, cudaMalloc(&L.gk, sizeof(float2) * c->NH), "lbfgs"));
    L.rho_host.assign(L.m, 0.0);
    return PMR_OK;
}

void lbfgs_free(pmr_ctx* c) {
    pmr::LBFGS& L = c->lb;
    for (double* p : {L.x, L.g, L.d, L.xt, L.gt, L.yk, L.S, L.Y, L.alpha}) cudaFree(p);
    cudaFree(L.gk);
    L = pmr::LBFGS{};
}

}  // namespace pmr
