// cs_action.cu -- Benincasa-Dowker action from the interval abundances
// (Section "The Benincasa-Dowker Action": Eqs. s2d_local, s3d_local,
// s4d_local, the smeared actions and the smearing functions f2, f3, f4).
//
// The local action is an exact integer bracket times a constant.  The
// smeared action sums N_k f(k, eps) over the whole histogram; those terms are
// orders of magnitude larger than the result (the thesis notes this for its
// de Sitter runs), so every term and the sum are carried in double-double
// arithmetic (FP64 error-free transformations), which keeps the cancellation
// far below a 1e-12 relative error at the largest N.
#include <cmath>

#include "cs_action.cuh"
#include "cs_kernels.cuh"
#include "cs_launch.cuh"

namespace cs {

namespace {

// Blocks of the smeared sum of cutoff kend with T threads each: one term per
// thread until kActBlocks blocks are full.
__host__ __device__ inline int act_blocks(int64_t kend, int T) {
    const int64_t b = (kend + T - 1) / T;
    return int(b < kActBlocks ? b : kActBlocks);
}

// Partial smeared sums, grid (blocks of the longest cutoff, eps).  GB300
// issues about two FP64 lanes per SM and cycle, and a term is a chain of
// FP64 operations: what bounds this is the chain's length and how few SMs
// the terms sit on.  So a block is one warp while the cutoffs are below 4096
// terms (wider beyond), the eps values run side by side, what does not
// depend on k comes from the host, and the sum is a shuffle tree.  256
// threads per block walking the eps values one after another took 102 us
// for n = 1024 .. 16384 and three smeared eps, squared powers per thread 19,
// powers from the host in one chain and the polynomial's products in eps all formed per
// term 16.8; this takes 11.4 (3+1 n = 16384: 13.0; with the final
// kernel's launch hidden behind it, a whole pass over a 2D order of 1024 lost 7 of 72 us).
struct ActPowers {
    EpsPowers e[kMaxEps];
    SmearCoef c[kMaxEps];
};
__global__ void __launch_bounds__(kActThreads) k_action_partial(int dim, const int64_t* __restrict__ hist,
                                                                EpsArgs eps, const __grid_constant__ ActPowers powers,
                                                                dd* __restrict__ partial) {
    __shared__ dd red[kActThreads / 32];
    const int e = blockIdx.y, T = blockDim.x, tid = threadIdx.x;
    const int64_t kend = eps.kend[e];  // 0 for a local action
    const int nb = act_blocks(kend, T);
    launch_dependents();  // k_action_final's launch, beside this one
    if (int(blockIdx.x) >= nb) return;
    dd sum = dd_from(0.0);
    for (int64_t k = int64_t(blockIdx.x) * T + tid; k < kend; k += int64_t(nb) * T) {
        const int64_t hk = hist[k];
        if (hk == 0) continue;
        sum = dd_add(sum, dd_times_i64(smear_term(dim, powers.c[e], powers.e[e], k), hk));
    }
    sum = warp_sum_dd(sum);
    if (T > 32) {  // uniform
        if ((tid & 31) == 0) red[tid >> 5] = sum;
        __syncthreads();
        if (tid < 32) sum = warp_sum_dd(tid < T / 32 ? red[tid] : dd_from(0.0));
    }
    if (tid == 0) partial[e * kActBlocks + blockIdx.x] = sum;
}

// One warp per eps: its partial sums, the action; warp 0 writes the bracket.
// After k_action_partial it is launched while that one runs, and waits here
// for its end (hist was complete before k_action_partial began).
__global__ void __launch_bounds__(32 * kMaxEps) k_action_final(int dim, int64_t n, const int64_t* hist,
                                                               int64_t len, EpsArgs eps, int T, const dd* partial,
                                                               double* out, int64_t* bracket) {
    const int e = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t h4[4] = {0, 0, 0, 0};
    for (int k = 0; k < 4 && k < len; ++k) h4[k] = hist[k];
    const int64_t b = bracket_of(dim, n, h4);
    const double ep = eps.v[e];
    wait_for_primary();
    if (threadIdx.x == 0 && bracket) *bracket = b;
    dd s;
    if (is_local(ep)) {
        s = local_action(eps.factor[e], b);
    } else {
        const int nb = act_blocks(eps.kend[e], T);
        dd sum = dd_from(0.0);
        for (int k = lane; k < nb; k += 32) sum = dd_add(sum, partial[e * kActBlocks + k]);
        s = smeared_action(dim, n, ep, eps.factor[e], warp_sum_dd(sum));
    }
    if (lane == 0) out[e] = s.hi + s.lo;
}

// B phi(j) from the layer sums (Eqs. b2d_local, b3d_local, b4d_local), one
// thread per element.
__global__ void k_dalembertian(int dim, int64_t n, const double* __restrict__ phi, const double* __restrict__ layer,
                               double scale, double* __restrict__ out) {
    for (int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; j < n; j += int64_t(gridDim.x) * blockDim.x) {
        const double p = phi ? phi[j] : 1.0;
        const double s0 = layer[j], s1 = layer[n + j], s2 = layer[2 * n + j];
        double b;
        if (dim == 2) {
            b = -p + 2.0 * (s0 - 2.0 * s1 + s2);
        } else if (dim == 3) {
            b = -p + s0 - 3.375 * s1 + 2.25 * s2;
        } else {
            const double s3 = layer[3 * n + j];
            b = -p + s0 - 9.0 * s1 + 16.0 * s2 - 8.0 * s3;
        }
        out[j] = scale * b;
    }
}

}  // namespace

cudaError_t launch_dalembertian(int dim, int64_t n, const double* phi, const double* layer, double ell, double* out,
                                cudaStream_t st) {
    const dd l2 = dd_two_prod(ell, ell);
    const dd c = dim == 2   ? dd_div(dd_from(2.0), l2)
                 : dim == 3 ? dd_div(dd_from(c3_const()), l2)
                            : dd_div(dd_from(4.0), dd_mul(l2, dd_sqrt(dd_from(6.0))));
    int64_t g = (n + 255) / 256;
    if (g > int64_t(device_sm_count()) * 8) g = int64_t(device_sm_count()) * 8;
    if (g < 1) g = 1;
    k_dalembertian<<<unsigned(g), 256, 0, st>>>(dim, n, phi, layer, c.hi + c.lo, out);
    return cudaGetLastError();
}

size_t action_workspace_bytes() { return sizeof(WsHeader) + size_t(kActBlocks) * kMaxEps * sizeof(dd); }

int action_host(int dim, int64_t n, const int64_t* hist, int64_t len, double eps, double* out, int64_t* bracket) {
    if (dim < 2 || dim > 4 || n < 0 || len < 0 || !(eps <= 1.0) || (len > 0 && !hist)) return CS_EINVAL;
    int64_t h4[4] = {0, 0, 0, 0};
    for (int k = 0; k < 4 && k < len; ++k) h4[k] = hist[k];
    const int64_t b = bracket_of(dim, n, h4);
    if (bracket) *bracket = b;
    dd s;
    if (is_local(eps)) {
        s = local_action(local_factor(dim), b);
    } else {
        const dd q = dd_two_sum(1.0, -eps);
        double R = 0.0;  // any histogram may come in here: bound by its own sum
        for (int64_t k = 0; k < len; ++k) R += fabs(double(hist[k]));
        const int64_t kend = smear_cutoff(dim, eps, R, len);
        dd sum = dd_from(0.0), p = dd_from(1.0);  // p = q^(max(0, k - deg))
        const int64_t deg = smear_deg(dim);
        for (int64_t k = 0; k < kend; ++k) {
            if (hist[k] != 0) sum = dd_add(sum, dd_mul(dd_from_i64(hist[k]), dd_mul(p, smear_poly(dim, k, q, eps))));
            if (k >= deg) p = dd_mul(p, q);
        }
        s = smeared_action(dim, n, eps, smeared_factor(dim, eps), sum);
    }
    if (out) *out = s.hi + s.lo;
    return CS_OK;
}

cudaError_t launch_action_device(int dim, int64_t n, const int64_t* hist, int64_t len, const double* eps, int n_eps,
                                 double* out, int64_t* bracket, void* workspace, cudaStream_t st) {
    EpsArgs a;
    a.n = n_eps;
    int64_t kmax = 0;
    for (int e = 0; e < kMaxEps; ++e) {
        a.v[e] = e < n_eps ? eps[e] : 0.0;
        a.kend[e] = is_local(a.v[e]) ? 0 : smear_cutoff(dim, a.v[e], 0.5 * double(n) * double(n), len);
        a.factor[e] = e < n_eps ? action_factor(dim, a.v[e]) : dd_from(0.0);
        kmax = a.kend[e] > kmax ? a.kend[e] : kmax;
    }
    int T = 32;  // threads per block: the fewest that give each thread one term
    while (T < kActThreads && kmax > int64_t(kActBlocks) * T) T *= 2;
    dd* partial = reinterpret_cast<dd*>(static_cast<uint8_t*>(workspace) + sizeof(WsHeader));
    if (kmax > 0) {
        ActPowers powers;
        for (int e = 0; e < kMaxEps; ++e)
            if (e < n_eps && !is_local(a.v[e])) {
                powers.e[e] = eps_powers(a.v[e]);
                powers.c[e] = smear_coef(dim, a.v[e]);
            }
        k_action_partial<<<dim3(unsigned(act_blocks(kmax, T)), unsigned(n_eps)), T, 0, st>>>(dim, hist, a, powers,
                                                                                          partial);
    }
    if (kmax == 0) {
        k_action_final<<<1, 32 * n_eps, 0, st>>>(dim, n, hist, len, a, T, partial, out, bracket);
        return cudaGetLastError();
    }
    return launch_after(k_action_final, dim3(1), unsigned(32 * n_eps), 0, st, dim, n, hist, len, a, T, partial, out,
                        bracket);
}

}  // namespace cs
