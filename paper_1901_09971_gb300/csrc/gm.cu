// Global-motion prior for RLOF tracking (arXiv 1901.09971, Section 3 "Parameters":
// RLOF with the global motion model, RLOF(IM-GM)). The paper prints no formula; the
// model used is a global affine motion fitted robustly to a sparse first pass and
// used as every point's initial flow in the main pass.
//
// The fit is an IRLS loop of a few iterations in one cooperative launch: the points form
// 64 parts, a CTA sums the weighted normal equations of one part in FP64 (GB300's FP64
// pipe is narrow, so the sums are spread over the SMs; of several parts, one after the
// other, where fewer than 64 CTAs are resident at once, as in a process that may use
// only some of the SMs) into the part's partial; the CTA that finishes last (a ticket
// counter) adds the partials in the parts' order, one thread per sum (deterministic, and
// the same bits for any number of CTAs), solves the two 3 x 3 systems and releases the
// others, which wait for it. The state (affine, fitted flag, go-on flag, ticket, released iteration) lives
// in the workspace, so no host round trip separates the stages: the main pass reads
// the fitted parameters from device memory.
//
// An iteration is a chain of FP64 latencies: sums, reduction, 64 additions, a solve of
// some dozen dependent divisions and square roots. With a launch an iteration, xor
// butterflies over all 13 sums and the two systems solved one after the other, the fit
// of 12,669 points took 8 x 23.3 us and the gaps between launches; in one launch, with
// halving exchanges and the systems solved in two lanes, 119 us. Same bits.
#include "common.cuh"
#include "batch.cuh"

namespace {

constexpr int kPartThreads = 256, kParts = 64;
constexpr unsigned kWaitTries = 1u << 24;  // polls (20 ns naps) before a CTA stops waiting for the last one
constexpr int kSums = 12;  // xx xy x yy y w | x qx, y qx, qx | x qy, y qy, qy

// Cholesky solve of the 3 x 3 normal equations (row-major m[9]); a pivot below
// 1e-10 of its diagonal entry counts as singular.
__device__ bool solve3(const double* m, const double* b, double* x)
{
    double L[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}}, z[3];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j <= i; ++j) {
            double s = m[3 * i + j];
            for (int k = 0; k < j; ++k) s -= L[i][k] * L[j][k];
            if (i == j) {
                if (!(s > 1e-10 * m[3 * i + i])) return false;
                L[i][i] = sqrt(s);
            } else {
                L[i][j] = s / L[j][j];
            }
        }
    for (int i = 0; i < 3; ++i) {
        double s = b[i];
        for (int k = 0; k < i; ++k) s -= L[i][k] * z[k];
        z[i] = s / L[i][i];
    }
    for (int i = 2; i >= 0; --i) {
        double s = z[i];
        for (int k = i + 1; k < 3; ++k) s -= L[k][i] * x[k];
        x[i] = s / L[i][i];
    }
    return true;
}

// State at the start of the workspace: a[6] (doubles), then int flags at byte 48
// (1 = fitted) and byte 52 (1 = iterating), the CTAs' ticket counter at byte 56 and the
// number of finished iterations at byte 60.
__global__ void gm_init_kernel(double* state)
{
    state[0] = 1; state[1] = 0; state[2] = 0;
    state[3] = 0; state[4] = 1; state[5] = 0;
    reinterpret_cast<int*>(state + 6)[0] = 0;
    reinterpret_cast<int*>(state + 6)[1] = 1;
    reinterpret_cast<unsigned*>(state + 7)[0] = 0;
    reinterpret_cast<unsigned*>(state + 7)[1] = 0;
}

// Sums of kSums + 1 values over the warp by halving exchanges: lanes 16 apart swap the
// halves of their values and add, then lanes 8 apart quarters, and so on; a lane ends
// with the total of value `lane / 2` (13 values padded to 16). Each total adds the lanes
// in the order of an xor butterfly, with 16 additions a lane instead of 65.
__device__ __forceinline__ double warp_totals(const double (&s)[kSums + 1])
{
    const int lane = threadIdx.x & 31;
    double v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = j <= kSums ? s[j] : 0.0;
#pragma unroll
    for (int o = 16, n = 8; o >= 2; o >>= 1, n >>= 1) {
        const bool hi = lane & o;
#pragma unroll
        for (int j = 0; j < n; ++j) {
            const double keep = hi ? v[n + j] : v[j], give = hi ? v[j] : v[n + j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// The IRLS iterations 0 .. iters - 1. Iteration k: sums over the points of part b, every
// kParts-th run of kPartThreads points (point i at pts[i * stride]); partial[b][0..11] =
// the 12 sums, [12] = the number of weighted points. The last CTA to finish adds the
// partials in the parts' order and solves the two 3 x 3 systems; a step with fewer than 3 weighted points
// or a singular matrix keeps the previous estimate and stops the loop. The waits are
// bounded: a CTA that gives up sets DGF_DEV_STAGE_WAIT and leaves (the others follow).
__global__ void __launch_bounds__(kPartThreads) gm_fit_kernel(const float* pts, int stride, const float* flow,
                                                              const uint8_t* status, int n, int iters, double c0,
                                                              double c_min, double* state, double* partial,
                                                              unsigned* dev_status)
{
    __shared__ double part[kPartThreads / 32][kSums + 1];
    __shared__ double tot[kSums + 1];
    __shared__ int last, go_on;
    int* flags = reinterpret_cast<int*>(state + 6);
    unsigned* ticket = reinterpret_cast<unsigned*>(state + 7);
    unsigned* done = ticket + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < iters; ++k) {
        double a[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) a[j] = __ldcg(state + j);
        const double ck = fmax(c_min, ldexp(c0, -(k - 1)));
        for (int b = blockIdx.x; b < kParts; b += gridDim.x) {
            double s[kSums + 1];
#pragma unroll
            for (int j = 0; j <= kSums; ++j) s[j] = 0.0;
            for (int i = b * kPartThreads + threadIdx.x; i < n; i += kParts * kPartThreads) {
                if (status[i] != DGF_TRACKED) continue;
                const float2 p = reinterpret_cast<const float2*>(pts)[(long long)i * stride];
                const float2 f = reinterpret_cast<const float2*>(flow)[i];
                const double x = p.x, y = p.y, qx = x + (double)f.x, qy = y + (double)f.y;
                double w = 1.0;
                if (k > 0) {
                    const double ex = a[0] * x + a[1] * y + a[2] - qx, ey = a[3] * x + a[4] * y + a[5] - qy;
                    const double e = sqrt(ex * ex + ey * ey);
                    if (e >= ck) continue;
                    const double u = 1.0 - (e / ck) * (e / ck);
                    w = u * u;
                }
                s[0] += w * x * x;
                s[1] += w * x * y;
                s[2] += w * x;
                s[3] += w * y * y;
                s[4] += w * y;
                s[5] += w;
                s[6] += w * x * qx;
                s[7] += w * y * qx;
                s[8] += w * qx;
                s[9] += w * x * qy;
                s[10] += w * y * qy;
                s[11] += w * qy;
                s[12] += 1.0;
            }
            // fixed-order reduction: over each warp, then one thread a sum over the warps
            const double v = warp_totals(s);
            __syncthreads();  // the part before has been read
            if (!(lane & 1) && lane / 2 <= kSums) part[warp][lane / 2] = v;
            __syncthreads();
            if (threadIdx.x <= kSums) {
                double t = 0.0;
                for (int w = 0; w < kPartThreads / 32; ++w) t += part[w][threadIdx.x];
                partial[b * (kSums + 1) + threadIdx.x] = t;
            }
        }
        if (threadIdx.x <= kSums) __threadfence();  // the partials are visible device-wide before this CTA's ticket
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == (unsigned)(k + 1) * gridDim.x - 1;
        __syncthreads();
        if (last) {
            // every other CTA's partial was written before its ticket
            __threadfence();
            if (threadIdx.x <= kSums) {
                double t = 0.0;
#pragma unroll 16
                for (int b = 0; b < kParts; ++b) t += __ldcg(partial + b * (kSums + 1) + threadIdx.x);
                tot[threadIdx.x] = t;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                // lanes 0 and 1 solve for the two rows of the affine at once
                const double m[9] = {tot[0], tot[1], tot[2], tot[1], tot[3], tot[4], tot[2], tot[4], tot[5]};
                const int r = lane & 1;
                const double rhs[3] = {tot[6 + 3 * r], tot[7 + 3 * r], tot[8 + 3 * r]};
                double x[3];
                const bool ok = __all_sync(0xffffffffu, !(tot[12] < 3.0) && solve3(m, rhs, x));
                if (ok && lane < 2) {
                    for (int j = 0; j < 3; ++j) state[3 * r + j] = x[j];
                    flags[0] = 1;
                }
                if (!ok && lane == 0) flags[1] = 0;  // keep the previous estimate
                __threadfence();
                __syncwarp();
                if (lane == 0) atomicExch(done, (unsigned)(k + 1));
            }
        }
        if (threadIdx.x == 0) {
            int ok = 0;
            for (unsigned i = 0; i < kWaitTries && !ok; ++i) {
                ok = *reinterpret_cast<volatile unsigned*>(done) >= (unsigned)(k + 1);
                if (!ok) __nanosleep(20);
            }
            __threadfence();
            if (!ok && dev_status) atomicOr(dev_status, (unsigned)DGF_DEV_STAGE_WAIT);
            go_on = ok && *reinterpret_cast<volatile int*>(flags + 1);
        }
        __syncthreads();
        if (!go_on) return;  // uniform: the fit has stopped
    }
}

bool gm_params_ok(const dgf_gm_params* g)
{
    return g && g->version == DGF_GM_PARAMS_VERSION && g->stride >= 1 && g->extra_levels >= 0 && g->iters >= 1 &&
           g->iters <= 64 && g->c0 > 0 && g->c_min > 0;
}

// Workspace layout: [a[6], flags, ticket; 256 B] [first-pass flow, n_sub x 8 B] [first-pass status, n_sub B]
// [the parts' partial sums, 64 x 13 doubles]
size_t flow_offset() { return 256; }
size_t status_offset(long long n_sub) { return dgf::round_up(flow_offset() + (size_t)n_sub * 8, 256); }
size_t partial_offset(long long n_sub) { return dgf::round_up(status_offset(n_sub) + (size_t)n_sub, 256); }
constexpr size_t kPartialBytes = (size_t)kParts * (kSums + 1) * 8;

}  // namespace

extern "C" void dgf_gm_params_default(dgf_gm_params* g)
{
    if (!g) return;
    g->version = DGF_GM_PARAMS_VERSION;
    g->stride = 4;
    g->extra_levels = 2;
    g->iters = 8;
    g->c0 = 32.0;
    g->c_min = 2.0;
}

extern "C" size_t dgf_gm_workspace(int n, const dgf_gm_params* g)
{
    if (n < 0 || !gm_params_ok(g)) return 0;
    const long long n_sub = ((long long)n + g->stride - 1) / g->stride;
    return dgf::round_up(partial_offset(n_sub) + kPartialBytes, 256);
}

extern "C" int rlof_track_gm(const void* pyr1, const void* pyr2, int W, int H, int pyr_levels, const float* pts, int n,
                             const dgf_rlof_params* p, const dgf_gm_params* g, float* flow, uint8_t* status,
                             uint8_t* iters, float* illum, void* workspace, size_t ws_bytes, cudaStream_t stream)
{
    dgf::TrackBatch main = {};
    int rc = dgf::prepare_params(p, main);
    if (rc != DGF_OK) return rc;
    if (!gm_params_ok(g) || n < 0 || W < 1 || H < 1 || pyr_levels > DGF_MAX_LEVELS ||
        pyr_levels < p->levels + g->extra_levels)
        return DGF_ERR_ARG;
    dgf_rlof_params deep = *p;
    deep.levels = p->levels + g->extra_levels;
    if ((rc = dgf::check_levels(W, H, &deep)) != DGF_OK) return rc;
    if (n == 0) return DGF_OK;
    if (!pyr1 || !pyr2 || !pts || !flow || !status || !workspace || !dgf::aligned(pyr1, 256) ||
        !dgf::aligned(pyr2, 256) || !dgf::aligned(pts, 8) || !dgf::aligned(flow, 8) ||
        (illum && !dgf::aligned(illum, 8)) || !dgf::aligned(workspace, 256))
        return DGF_ERR_ARG;
    if (ws_bytes < dgf_gm_workspace(n, g)) return DGF_ERR_WORKSPACE;
    const long long n_sub = ((long long)n + g->stride - 1) / g->stride;
    char* ws = static_cast<char*>(workspace);
    double* affine = reinterpret_cast<double*>(ws);
    float* sub_flow = reinterpret_cast<float*>(ws + flow_offset());
    uint8_t* sub_status = reinterpret_cast<uint8_t*>(ws + status_offset(n_sub));

    // 1. sparse first pass with the deeper pyramid (deep.levels <= pyr_levels <= DGF_MAX_LEVELS)
    dgf::TrackBatch first = {};
    if ((rc = dgf::prepare_params(&deep, first)) != DGF_OK) return rc;
    first.pyr_levels = pyr_levels;
    first.n_jobs = 1;
    first.total = (int)n_sub;
    first.jobs[0] = dgf::TrackJob{static_cast<const char*>(pyr1), static_cast<const char*>(pyr2), W, H, pts, sub_flow,
                                  sub_status, nullptr, nullptr, 0, g->stride, nullptr};
    if ((rc = dgf::launch_track(first, &deep, stream)) != DGF_OK) return rc;
    // 2. robust affine fit
    double* partial = reinterpret_cast<double*>(ws + partial_offset(n_sub));
    unsigned* dev_status = dgf::status_word();  // (null: the kernel records nothing)
    gm_init_kernel<<<1, 1, 0, stream>>>(affine);
    {
        int n_pts = (int)n_sub, stride = g->stride, iters = g->iters;
        double c0 = g->c0, c_min = g->c_min;
        void* args[] = {(void*)&pts, (void*)&stride, (void*)&sub_flow, (void*)&sub_status, (void*)&n_pts, (void*)&iters,
                        (void*)&c0, (void*)&c_min, (void*)&affine, (void*)&partial, (void*)&dev_status};
        const unsigned grid = dgf::cooperative_blocks(gm_fit_kernel, kPartThreads, kParts);
        if ((rc = dgf::launch_cooperative((const void*)gm_fit_kernel, grid, dim3(kPartThreads), args, stream)) != DGF_OK)
            return rc;
    }
    // 3. main pass from the prior
    main.pyr_levels = pyr_levels;
    main.n_jobs = 1;
    main.total = n;
    main.jobs[0] = dgf::TrackJob{static_cast<const char*>(pyr1), static_cast<const char*>(pyr2), W, H, pts, flow, status,
                                 iters, illum, 0, 1, affine};
    return dgf::launch_track(main, p, stream);
}
