// logdet.cu -- log|A| (Sec. 3; the method is left open in Sec. 4.6 / App. B.7):
//   * SLQ: stochastic Lanczos quadrature (Ubaru, Chen & Saad 2017) on Ah = D^{-1/2} A D^{-1/2}.
//     For every probe z_s the tridiagonal T_s comes from the recorded CG coefficients (CG-Lanczos
//     relation), and log|Ah| ~= (n/m) sum_s sum_j tau_sj^2 log theta_sj with T_s's eigenvalues theta_j
//     and eigenvector first components tau_j; the inner sum e_1^T log(T_s) e_1 is evaluated without
//     them, by the trapezoidal rule on an integral of the logarithm, in FP64.
//   * EXACT: FP64 Cholesky of Ah by tiles (cholesky.cu), log|Ah| = 2 sum log L_ii and the y solve.
//   log|A| = sum log D_ii + log|Ah| in both cases.
#include <cmath>
#include <cstring>
#include <mutex>

#include "gp2s_cholesky.cuh"
#include "gp2s_internal.cuh"
#include "gp2s_kernel_math.cuh"

namespace gp2s {

namespace {

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------------------------------------
// Gauss quadrature of the logarithm of one probe's tridiagonal T (k x k, positive definite):
//     e_1^T log(T) e_1 = sum_j tau_j^2 log theta_j
// without its eigen-decomposition, from log(x) = int_0^inf (1 / (1 + t) - 1 / (x + t)) dt.  With t = e^u
// the integrand is analytic in the strip |Im u| < pi (its poles are t = -1 and t = -theta_j) and
// decays like e^-|u|, so the trapezoidal rule with step h converges like e^(-2 pi^2 / h): h = 1/2
// gives 7e-18.  Each node needs g(t) = e_1^T (T + t I)^{-1} e_1, the continued fraction
// f_j = a_j + t - b_j^2 / f_{j+1}, g = 1 / f_0, all of whose pivots are positive for a positive
// definite T (a pivot that is not, reports one).  The nodes run from t = 3e-30 (below the rounding
// of any diagonal entry) to e^40 times Gershgorin's bound: about 220 of them, one thread each.
//
// What bounds it: the chain of k divisions per node, 256 nodes wide, on the FP64 pipe (one
// sixty-fourth of the FP32 rate).  The implicit QR iteration that it replaces ran about 1.7 k^2 / 2
// rotations one after the other in one thread: at k = 100 it took 24 to 90 ms for 64 probes.
// Measured
// around it: the log-determinant of 200,003 points in 2-D (64 probes) 112.8 -> 26.9 ms, a batch of 24
// problems (16 probes) 812 -> 453 ms, the results equal to 3e-16.
// ---------------------------------------------------------------------------------------------
constexpr int kSlqThreads = 256;
constexpr int kSlqFirst = -136;          // first node, u = kSlqFirst h
constexpr double kSlqStep = 0.5;         // h

// One CTA per probe: T from the recorded CG coefficients, then the quadrature nodes.
__global__ void __launch_bounds__(kSlqThreads)
k_slq(const double *__restrict__ rec, const double *__restrict__ sc, int m, int ksteps, double *__restrict__ out,
      int *__restrict__ bad)
{
    extern __shared__ double slq_sh[];
    __shared__ double red[kSlqThreads / 32];
    __shared__ int flag;
    const int s = blockIdx.x;
    if (s >= m) return;
    double *a = slq_sh;                  // diagonal
    double *b2 = a + ksteps;             // squared off-diagonals
    // number of recorded steps for this probe column (column s + 1 of the CG scalar block)
    const int steps = (int)sc[(s + 1) * kScal + S_STEPS];
    const int k = steps < ksteps ? steps : ksteps;
    if (k <= 0) {
        if (threadIdx.x == 0) {
            out[s] = 0.0;
            atomicOr(bad, 1);
        }
        return;
    }
    if (threadIdx.x == 0) flag = 0;
    __syncthreads();
    const double *al = rec + (int64_t)s * ksteps * 2;
    // CG-Lanczos relation: T_00 = 1/alpha_0; T_jj = 1/alpha_j + beta_{j-1}/alpha_{j-1};
    // T_{j,j+1}^2 = beta_j/alpha_j^2
    for (int j = threadIdx.x; j < k; j += kSlqThreads) {
        const double aj = al[2 * j];
        a[j] = 1.0 / aj + (j > 0 ? al[2 * (j - 1) + 1] / al[2 * (j - 1)] : 0.0);
        b2[j] = j + 1 < k ? al[2 * j + 1] / (aj * aj) : 0.0;
        if (!(b2[j] >= 0.0)) atomicOr(&flag, 2);
    }
    __syncthreads();
    // Gershgorin's bound on the largest Ritz value
    double r = 1.0;
    for (int j = threadIdx.x; j < k; j += kSlqThreads)
        r = fmax(r, a[j] + (j > 0 ? sqrt(b2[j - 1]) : 0.0) + sqrt(b2[j]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = fmax(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = r;
    __syncthreads();
    r = red[0];
#pragma unroll
    for (int w = 1; w < kSlqThreads / 32; ++w) r = fmax(r, red[w]);
    // a bound that is not finite comes from coefficients that are not: no quadrature
    const bool fin = isfinite(r);
    const int last = fin ? (int)ceil((40.0 + log(r)) / kSlqStep) : kSlqFirst - 1;
    double g = 0.0;
    bool pos = fin;
    for (int i = kSlqFirst + (int)threadIdx.x; i <= last; i += kSlqThreads) {
        const double t = exp(kSlqStep * i);
        double f = a[k - 1] + t;
        pos = pos && f > 0.0;
        for (int j = k - 2; j >= 0; --j) {
            f = (a[j] + t) - b2[j] / f;
            pos = pos && f > 0.0;
        }
        g += t / (1.0 + t) - t / f;
    }
    if (!pos) atomicOr(&flag, 4);
    g = warp_sum_d(g);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = g;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < kSlqThreads / 32; ++w) v += red[w];
        if (flag) atomicOr(bad, flag);
        out[s] = flag ? nan("") : kSlqStep * v;
    }
}

__global__ void k_sum_log(const double *__restrict__ D, int64_t n, double *__restrict__ part)
{
    __shared__ double sh[32];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += log(D[i]);
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

__global__ void k_dot64(const double *__restrict__ a, const double *__restrict__ b, int64_t n,
                        double *__restrict__ part)
{
    __shared__ double sh[32];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s = fma(a[i], b[i], s);
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

gp2s_status reduce_parts(gp2s_ctx *c, const double *part, int cnt, double *out_host)
{
    std::vector<double> h(cnt);
    GP2S_CUDA(c, cudaMemcpyAsync(h.data(), part, sizeof(double) * cnt, cudaMemcpyDeviceToHost, c->stream));
    GP2S_CUDA(c, cudaStreamSynchronize(c->stream));
    double s = 0.0;
    for (int k = 0; k < cnt; ++k) s += h[k];
    *out_host = s;
    return GP2S_OK;
}

}  // namespace

gp2s_status sum_log_diag(gp2s_ctx *c, double *out_host)
{
    const int nb = 152 * 2;
    GP2S_TRY(ensure(c, c->gpart, sizeof(double) * (2 * nb + 8)));
    k_sum_log<<<nb, 256, 0, c->stream>>>(c->D64.as<double>(), c->A.n, c->gpart.as<double>());
    GP2S_LAUNCH(c);
    return reduce_parts(c, c->gpart.as<double>(), nb, out_host);
}

gp2s_status dot_f64(gp2s_ctx *c, const double *a, const double *b, int64_t n, double *out_host)
{
    const int nb = 152 * 2;
    GP2S_TRY(ensure(c, c->gpart, sizeof(double) * (2 * nb + 8)));
    k_dot64<<<nb, 256, 0, c->stream>>>(a, b, n, c->gpart.as<double>());
    GP2S_LAUNCH(c);
    return reduce_parts(c, c->gpart.as<double>(), nb, out_host);
}

// SLQ scratch: the m quadratures, the failure flag, and a snapshot of the CG scalar block (the step
// counts k_slq reads) taken when the launch is queued.
static void slq_layout(gp2s_ctx *c, int m, double **out, int **bad, double **snap)
{
    *out = c->slq_work.as<double>();
    *bad = reinterpret_cast<int *>(*out + m);
    *snap = *out + m + 8;
}

static gp2s_status slq_launch(gp2s_ctx *c, cudaStream_t wait_on, cudaStream_t run_on, int m, int ksteps)
{
    GP2S_TRY(ensure(c, c->slq_work, sizeof(double) * ((size_t)m + 8 + (size_t)kScal * (m + 1)) + 64));
    double *out, *snap;
    int *bad;
    slq_layout(c, m, &out, &bad, &snap);
    GP2S_CUDA(c, cudaMemcpyAsync(snap, c->scal.as<double>(), sizeof(double) * kScal * (m + 1), cudaMemcpyDeviceToDevice,
                                 wait_on));
    GP2S_CUDA(c, cudaMemsetAsync(bad, 0, sizeof(int), wait_on));
    if (run_on != wait_on) {
        GP2S_CUDA(c, cudaEventRecord(c->slq_ev_rec, wait_on));
        GP2S_CUDA(c, cudaStreamWaitEvent(run_on, c->slq_ev_rec, 0));
    }
    const size_t smem = sizeof(double) * 2 * (size_t)ksteps;
    GP2S_TRY(smem_attr(c, (const void *)k_slq, smem));
    k_slq<<<m, kSlqThreads, smem, run_on>>>(c->rec.as<double>(), snap, m, ksteps, out, bad);
    GP2S_LAUNCH(c);
    return GP2S_OK;
}

gp2s_status slq_start_async(gp2s_ctx *c, int m, int ksteps)
{
    if (!c->side_stream) {
        GP2S_CUDA(c, cudaStreamCreateWithFlags(&c->side_stream, cudaStreamNonBlocking));
        GP2S_CUDA(c, cudaEventCreateWithFlags(&c->slq_ev_rec, cudaEventDisableTiming));
        GP2S_CUDA(c, cudaEventCreateWithFlags(&c->slq_ev_done, cudaEventDisableTiming));
    }
    GP2S_TRY(slq_fence(c));
    GP2S_TRY(slq_launch(c, c->stream, c->side_stream, m, ksteps));
    GP2S_CUDA(c, cudaEventRecord(c->slq_ev_done, c->side_stream));
    c->slq_pending = true;
    c->slq_m = m;
    c->slq_k = ksteps;
    return GP2S_OK;
}

gp2s_status slq_fence(gp2s_ctx *c)
{
    if (c->slq_pending) GP2S_CUDA(c, cudaStreamWaitEvent(c->stream, c->slq_ev_done, 0));
    return GP2S_OK;
}

gp2s_status slq_logdet(gp2s_ctx *c, int m, int ksteps, double *logdet_hat, double *stderr_hat)
{
    if (m <= 0 || !c->have_probes) return set_err(c, GP2S_ENOTREADY, "SLQ needs the probe CG run");
    if (c->slq_pending && c->slq_m == m && c->slq_k == ksteps) {
        GP2S_TRY(slq_fence(c));   // queued beside the probe solves, from the same recorded steps
    } else {
        GP2S_TRY(slq_fence(c));
        GP2S_TRY(slq_launch(c, c->stream, c->stream, m, ksteps));
    }
    c->slq_pending = false;
    double *out, *snap;
    int *bad;
    slq_layout(c, m, &out, &bad, &snap);
    std::vector<double> g(m);
    int hbad = 0;
    GP2S_CUDA(c, cudaMemcpyAsync(g.data(), out, sizeof(double) * m, cudaMemcpyDeviceToHost, c->stream));
    GP2S_CUDA(c, cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    GP2S_CUDA(c, cudaStreamSynchronize(c->stream));
    if (hbad) return set_err(c, GP2S_EBREAKDOWN, "SLQ: a tridiagonal is not positive definite or not finite");
    const double n = (double)c->A.n;
    double mean = 0.0;
    for (int s = 0; s < m; ++s) mean += n * g[s];
    mean /= m;
    double var = 0.0;
    for (int s = 0; s < m; ++s) var += (n * g[s] - mean) * (n * g[s] - mean);
    var = m > 1 ? var / (m - 1) : 0.0;
    *logdet_hat = mean;
    if (stderr_hat) *stderr_hat = std::sqrt(var / m);
    return GP2S_OK;
}

}  // namespace gp2s

// =============================================================================================
// Allocation-free exact LML for small problems (gp2s_lml_exact_noalloc).
//
// For callers that may not allocate device memory (work issued during CUDA stream capture, or a
// device whose memory is owned by another allocator), every intermediate of this path lives in one
// fixed array compiled into the library.  The dense matrix is built pair by pair with the same
// exact FP64 support test and FP64 kernel value as the CSR path, then factored by the same tiled
// Cholesky kernel as the EXACT log-determinant (cholesky.cu), with every tile present.
// =============================================================================================
namespace gp2s {

namespace {

constexpr int kNoAllocMaxN = GP2S_NOALLOC_MAX_N;
constexpr int kNoAllocNT = kNoAllocMaxN / kCT;                                   // tile rows
constexpr int kNoAllocTiles = kNoAllocNT * (kNoAllocNT + 1) / 2;
constexpr size_t kNoAllocVec = (size_t)kNoAllocTiles * kCTElems;                 // 1 / diag(L), y', x', a (4 n)
constexpr size_t kNoAllocB = kNoAllocVec + 4 * kNoAllocMaxN;                     // bump table n x L
constexpr size_t kNoAllocFlag = kNoAllocB + (size_t)kNoAllocMaxN * kMaxBumps;    // tile flags and the pivot flag (int)
constexpr size_t kNoAllocDoubles = kNoAllocFlag + 128;
static_assert(kNoAllocMaxN % kCT == 0 && kNoAllocTiles + 2 * kNoAllocNT + 3 <= 256, "the flags fit their place");

// The scratch array: every call on a device shares it (about 1.3 MB per device).
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

std::mutex g_noalloc_mu;
double *g_noalloc_ptr[64] = {};   // device address of g_noalloc_scratch per device ordinal

template <int D>
__global__ void k_noalloc_bumps(const double *__restrict__ X, int n, KernelParams kp, double *__restrict__ B)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int l = 0; l < kp.L; ++l) {
        double q = 0.0;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            double dk = X[(int64_t)i * D + k] - kp.centers[l * D + k];
            q = q + dk * dk;
        }
        double rho = kp.radii[l];
        double s = q / (rho * rho);
        double e = s < 1.0 ? exp(kp.beta * (1.0 - 1.0 / (1.0 - s))) : 0.0;
        B[(int64_t)i * kp.L + l] = kp.amps[l] * e;
    }
}

// Slot of tile (i, j), i >= j, of the packed lower triangle of nt x nt tiles (columns one after the other).
__host__ __device__ inline int noalloc_slot(int nt, int i, int j) { return j * nt - j * (j - 1) / 2 + (i - j); }

// The lower triangle of A = K + sigma2 I in tiles, rows past n as identity rows (every element is
// written, so no clearing is needed).  One CTA per tile.
template <int D>
__global__ void k_noalloc_tiles(const double *__restrict__ X, int n, int nt, KernelParams kp,
                                const double *__restrict__ B, double *__restrict__ tiles)
{
    int tj = 0, at = blockIdx.x;
    while (at >= nt - tj) {
        at -= nt - tj;
        ++tj;
    }
    const int ti = tj + at;
    for (int e = threadIdx.x; e < kCTElems; e += blockDim.x) {
        const int i = ti * kCT + e / kCT, j = tj * kCT + e % kCT;
        double v = i == j ? 1.0 : 0.0;
        if (i < n && j <= i) {
            double q = 0.0;
#pragma unroll
            for (int k = 0; k < D; ++k) {
                double dk = __dsub_rn(X[(int64_t)i * D + k], X[(int64_t)j * D + k]);
                q = __dadd_rn(q, __dmul_rn(dk, dk));
            }
            v = 0.0;
            if (i == j || q < kp.r * kp.r) {
                double S = 0.0;
                for (int l = 0; l < kp.L; ++l) S = fma(B[(int64_t)i * kp.L + l], B[(int64_t)j * kp.L + l], S);
                v = wendland<double>(kp.kind, D, sqrt(q) * kp.inv_r) * (S + kp.w0);
                if (i == j) v += kp.sigma2;
            }
        }
        tiles[(size_t)blockIdx.x * kCTElems + e] = v;
    }
}

// {LML, y^T a, log|A|} from the factor's diagonal and the solution; NaN when a pivot failed.
__global__ void k_noalloc_finish(const double *__restrict__ tiles, int n, int nt, const double *__restrict__ y,
                                 const double *__restrict__ a, const int *__restrict__ bad, double *__restrict__ out)
{
    __shared__ double sh[2][32];
    double ld = 0.0, qd = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int j = i / kCT, r = i % kCT;
        ld += log(tiles[(size_t)noalloc_slot(nt, j, j) * kCTElems + r * kCT + r]);
        qd = fma(y[i], a[i], qd);
    }
    ld = warp_sum_d(ld);
    qd = warp_sum_d(qd);
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = ld;
        sh[1][threadIdx.x >> 5] = qd;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double L2 = 0.0, Q = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { L2 += sh[0][w]; Q += sh[1][w]; }
        double logdet = 2.0 * L2;
        double lml = -0.5 * Q - 0.5 * logdet - 0.5 * (double)n * log(2.0 * 3.141592653589793);
        if (*bad) { lml = nan(""); Q = nan(""); logdet = nan(""); }
        out[0] = lml;
        out[1] = Q;
        out[2] = logdet;
    }
}

// Device address of the scratch array on the current device, looked up once per device.
gp2s_status noalloc_scratch(double **ptr)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return GP2S_ECUDA; }
    if (dev < 0 || dev >= 64) return GP2S_ECUDA;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) { cudaGetLastError(); return GP2S_ECUDA; }
        g_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *ptr = g_noalloc_ptr[dev];
    return GP2S_OK;
}

template <int D>
void launch_noalloc_build(const double *X, int n, int nt, const KernelParams &kp, double *B, double *tiles, cudaStream_t s)
{
    k_noalloc_bumps<D><<<(n + 127) / 128, 128, 0, s>>>(X, n, kp, B);
    k_noalloc_tiles<D><<<chol_dense_tiles(nt), 256, 0, s>>>(X, n, nt, kp, B, tiles);
}

}  // namespace

gp2s_status validate_hyper(gp2s_ctx *c, const gp2s_hyper *h);   // assemble.cu
KernelParams make_kernel_params(const gp2s_hyper *h);             // assemble.cu

}  // namespace gp2s

extern "C" gp2s_status gp2s_lml_exact_noalloc(int64_t n, const double *X_dev, const double *y_dev,
                                              const gp2s_hyper *hyper, double *out_dev, void *cuda_stream)
{
    using namespace gp2s;
    if (n < 1 || n > kNoAllocMaxN) return GP2S_EINVAL;
    if (!X_dev || !y_dev || !out_dev) return GP2S_EINVAL;
    if (validate_hyper(nullptr, hyper) != GP2S_OK) return GP2S_EINVAL;
    if (hyper->family != GP2S_KERNEL_PRODUCT) return GP2S_EINVAL;   // the product kernel only
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    // the scratch address is per device: a stream of another device would get this device's
    // address, so such a stream is refused (the legacy and per-thread default streams follow the
    // current device).  The stream's device is not asked for while the stream is being captured,
    // where that query invalidates the capture: a capture records on the stream's own device, and
    // the caller answers for the device being current.
    if (s != nullptr && s != cudaStreamLegacy && s != cudaStreamPerThread) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) {
            cudaGetLastError();
            return GP2S_ECUDA;
        }
        if (cs == cudaStreamCaptureStatusNone) {
            int cur = 0, sdev = 0;
            if (cudaGetDevice(&cur) != cudaSuccess || cudaStreamGetDevice(s, &sdev) != cudaSuccess) {
                cudaGetLastError();
                return GP2S_ECUDA;
            }
            if (sdev != cur) return GP2S_EINVAL;
        }
    }
    double *base = nullptr;
    gp2s_status st = noalloc_scratch(&base);
    if (st != GP2S_OK) return st;
    const int nn = (int)n;
    const KernelParams kp = make_kernel_params(hyper);
    // A's tiles, factored in place; a = A^{-1} y in the last of the four vectors
    CholArgs ca{};
    ca.nt = (nn + kCT - 1) / kCT;
    ca.ntiles = chol_dense_tiles(ca.nt);
    ca.ntasks = ca.ntiles + 2 * ca.nt;
    ca.n = nn;
    ca.last = ca.nt - 1;
    ca.solve = 1;
    ca.tiles = base;
    ca.dinv = base + kNoAllocVec;
    ca.yv = ca.dinv + kNoAllocMaxN;
    ca.xv = ca.yv + kNoAllocMaxN;
    ca.x = ca.xv + kNoAllocMaxN;
    ca.b = y_dev;
    ca.flags = reinterpret_cast<int *>(base + kNoAllocFlag);
    const size_t flags = chol_flag_ints(ca.ntiles, ca.nt);
    ca.bad = ca.flags + flags;
    double *B = base + kNoAllocB;
    if (cudaMemsetAsync(ca.flags, 0, sizeof(int) * (flags + 1), s) != cudaSuccess) { cudaGetLastError(); return GP2S_ECUDA; }
    switch (hyper->d) {
    case 1: launch_noalloc_build<1>(X_dev, nn, ca.nt, kp, B, ca.tiles, s); break;
    case 2: launch_noalloc_build<2>(X_dev, nn, ca.nt, kp, B, ca.tiles, s); break;
    case 3: launch_noalloc_build<3>(X_dev, nn, ca.nt, kp, B, ca.tiles, s); break;
    default: launch_noalloc_build<4>(X_dev, nn, ca.nt, kp, B, ca.tiles, s); break;
    }
    if (chol_launch(ca, 152, s) != cudaSuccess) return GP2S_ECUDA;
    k_noalloc_finish<<<1, 256, 0, s>>>(ca.tiles, nn, ca.nt, y_dev, ca.x, ca.bad, out_dev);
    if (cudaGetLastError() != cudaSuccess) return GP2S_ECUDA;
    return GP2S_OK;
}
