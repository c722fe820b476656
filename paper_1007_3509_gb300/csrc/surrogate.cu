// Training data for the learned field surrogate, generated by the Monte Carlo
// crystal plasticity itself (Sec. 2), and the per-grain driving field the
// trained network produces.
//
// Orientation encoding: the Taylor strain of Eq. (3) is axisymmetric about
// the sample x axis, so a crystal's response depends on its orientation only
// through the loading axis d = R^T e_x, and only modulo the cubic symmetry of
// the crystal.  The network therefore sees four cubic invariants of d instead
// of the raw quaternion (which also carries the irrelevant rotation about x
// and the q/-q double cover): |d| sorted in decreasing order (3) and
// d1^2 d2^2 + d2^2 d3^2 + d3^2 d1^2 (1).
//
// Data: n_orient orientations, each followed through n_incr Taylor load
// increments (Eq. (3)) in K independent stochastic histories (K material
// points per orientation, different Philox counters).  After increment t the
// population-average sample-frame stress sigma_hat(t) = <R sigma_c R^T> and
// slip gamma_hat(t) = <gamma> are reduced over all points, and every
// orientation o contributes one sample
//   x = (f(q_o), sigma_hat(t) / stress_scale, gamma_hat(t) / strain_scale)
//   y = (<w>_K / w_scale, <E_rho>_K / erho_scale)
// with <.>_K the average over the orientation's K histories.
// Field: for every grain g, y = MLP(f(q_g), load state) and
//   b_g = round-half-even(256 energy_scale (y0 w_scale + y1 erho_scale)),
// clamped to +-2^20, the per-grain table of HP_FIELD_GRAIN.
#include <math.h>

#include <vector>

#include "common.cuh"

namespace hp {
namespace {

constexpr int kT = 256;

__global__ void k_point_grain(int64_t P, int32_t K, int32_t* grain) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < P) grain[p] = (int32_t)(p / K);
}

// acc[0..5] += sample-frame stress, acc[6] += gamma (FP64 accumulation)
__global__ void k_load_reduce(int64_t P, const int32_t* grain, const float* quat, const float* sigma,
                              const float* gamma, double* acc) {
    __shared__ double part[7][kT / 32];
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double v[7] = {0, 0, 0, 0, 0, 0, 0};
    if (p < P) {
        const float* q = quat + 4 * (int64_t)grain[p];
        const double n = sqrt((double)q[0] * q[0] + (double)q[1] * q[1] + (double)q[2] * q[2] + (double)q[3] * q[3]);
        const double w = q[0] / n, x = q[1] / n, y = q[2] / n, z = q[3] / n;
        const double R[3][3] = {{1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)},
                                {2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)},
                                {2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)}};
        double s[3][3];
        const float s0 = sigma[p], s1 = sigma[P + p], s2 = sigma[2 * P + p], s3 = sigma[3 * P + p],
                    s4 = sigma[4 * P + p], s5 = sigma[5 * P + p];
        s[0][0] = s0; s[1][1] = s1; s[2][2] = s2;
        s[1][2] = s[2][1] = s3; s[0][2] = s[2][0] = s4; s[0][1] = s[1][0] = s5;
        const int I[6] = {0, 1, 2, 1, 0, 0}, J[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            double a = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int l = 0; l < 3; ++l) a += R[I[c]][k] * s[k][l] * R[J[c]][l];
            v[c] = a;
        }
        v[6] = gamma[p];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 7; ++c) {
        double a = v[c];
        for (int m = 16; m >= 1; m >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, m);
        if (lane == 0) part[c][wid] = a;
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        double a = 0.0;
        for (int i = 0; i < kT / 32; ++i) a += part[threadIdx.x][i];
        atomicAdd(acc + threadIdx.x, a);
    }
}

struct Scales {
    float stress, strain, w, erho;
};

// Writes row o * row_stride of X and Y (row_stride = n_incr, X and Y offset to the increment).
__global__ void k_collect(int32_t n_orient, int32_t K, const float* quat, const float* w, const float* erho,
                          const double* acc, double inv_p, Scales sc, int32_t row_stride, float* X, float* Y) {
    const int32_t o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n_orient) return;
    double sw = 0.0, se = 0.0;
    for (int h = 0; h < K; ++h) {
        sw += w[(int64_t)o * K + h];
        se += erho[(int64_t)o * K + h];
    }
    const int64_t row = (int64_t)o * row_stride;
    float* x = X + row * 11;
    orient_features(quat + 4 * (int64_t)o, x);
#pragma unroll
    for (int c = 0; c < 6; ++c) x[4 + c] = (float)(acc[c] * inv_p / sc.stress);
    x[10] = (float)(acc[6] * inv_p / sc.strain);
    Y[2 * row + 0] = (float)(sw / K / sc.w);
    Y[2 * row + 1] = (float)(se / K / sc.erho);
}

__global__ void k_load_out(const double* acc, double inv_p, float* out) {
    if (threadIdx.x < 7) out[threadIdx.x] = (float)(acc[threadIdx.x] * inv_p);
}

}  // namespace
}  // namespace hp

using namespace hp;


extern "C" int hp_sur_generate(const hp_cp_params* prm, uint64_t seed, const float* quat, int32_t n_orient, int32_t K,
                               int32_t n_incr, const hp_sur_scales* sc, float* X, float* Y, float* load_out,
                               void* stream) {
    hp::Range r_("hp_sur_generate");
    if (!prm || !quat || n_orient < 1 || K < 1 || n_incr < 1 || !sc || !X || !Y)
        return set_error(HP_ERR_ARG, "hp_sur_generate: bad arguments");
    cudaStream_t s = as_stream(stream);
    const int64_t P = (int64_t)n_orient * K;
    float *eps = nullptr, *gam = nullptr, *g = nullptr, *sig = nullptr, *w = nullptr, *er = nullptr;
    int32_t* grain = nullptr;
    double* acc = nullptr;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void** p, size_t bytes) { if (e == cudaSuccess) e = cudaMallocAsync(p, bytes, s); };
    alloc((void**)&eps, sizeof(float) * 6 * P);
    alloc((void**)&gam, sizeof(float) * P);
    alloc((void**)&g, sizeof(float) * P);
    alloc((void**)&sig, sizeof(float) * 6 * P);
    alloc((void**)&w, sizeof(float) * P);
    alloc((void**)&er, sizeof(float) * P);
    alloc((void**)&grain, sizeof(int32_t) * P);
    alloc((void**)&acc, sizeof(double) * 8 * n_incr);
    int rc = HP_OK;
    if (e != cudaSuccess) rc = set_error(HP_ERR_OOM, "hp_sur_generate: allocation failed");
    Scales scl{sc->stress, sc->strain, sc->w, sc->erho};
    if (rc == HP_OK) {
        const unsigned pb = (unsigned)((P + kT - 1) / kT);
        ::hp::count_launch();
        k_point_grain<<<pb, kT, 0, s>>>(P, K, grain);
        cudaMemsetAsync(acc, 0, sizeof(double) * 8 * n_incr, s);
        hp_cp_state st{P, eps, gam, g};
        rc = hp_cp_reset(prm, &st, s);
        for (int32_t t = 1; t <= n_incr && rc == HP_OK; ++t) {
            rc = hp_cp_step(prm, seed, grain, quat, (uint32_t)(t - 1), 1, &st, sig, w, er, nullptr, s);
            if (rc) break;
            double* a = acc + 8 * (t - 1);
            ::hp::count_launch();
            k_load_reduce<<<pb, kT, 0, s>>>(P, grain, quat, sig, gam, a);
            ::hp::count_launch();
            k_collect<<<(n_orient + kT - 1) / kT, kT, 0, s>>>(n_orient, K, quat, w, er, a, 1.0 / (double)P, scl, n_incr,
                                                              X + (int64_t)(t - 1) * 11, Y + (int64_t)(t - 1) * 2);
            if (load_out) {
                ::hp::count_launch();
                k_load_out<<<1, 32, 0, s>>>(a, 1.0 / (double)P, load_out + 7 * (t - 1));
            }
        }
        if (rc == HP_OK && (e = cudaGetLastError()) != cudaSuccess) rc = cuda_error(e, "hp_sur_generate");
    }
    cudaFreeAsync(eps, s); cudaFreeAsync(gam, s); cudaFreeAsync(g, s); cudaFreeAsync(sig, s);
    cudaFreeAsync(w, s); cudaFreeAsync(er, s); cudaFreeAsync(grain, s); cudaFreeAsync(acc, s);
    return rc;
}

extern "C" int hp_sur_field(const float* params, const float* quat, int32_t G, const float* load,
                            const hp_sur_scales* sc, double energy_scale, int32_t* b_out, float* e_out, void* stream) {
    if (!params || !quat || G < 1 || !load || !sc || !b_out) return set_error(HP_ERR_ARG, "hp_sur_field: bad arguments");
    FieldIO io;
    io.quat = quat;
    for (int c = 0; c < 7; ++c) io.load[c] = load[c];  // copied into the launch: the caller may free load
    io.stress = sc->stress;
    io.strain = sc->strain;
    io.w = sc->w;
    io.erho = sc->erho;
    io.scale = (float)energy_scale;
    io.b = b_out;
    io.e = e_out;
    return mlp_field(params, io, G, as_stream(stream));
}

extern "C" int hp_sur_train(float* params, float* m, float* v, const float* X, const float* Y, int64_t M,
                            const hp_sur_train_params* tp, int32_t step0, float* loss, float* loss_log, void* stream) {
    hp::Range r_("hp_sur_train");
    if (!params || !m || !v || !X || !Y || M < 1 || !tp || step0 < 0 || tp->steps < 0 || tp->group < 1 ||
        tp->batch < 0 || !(tp->lr > 0.0f) || !(tp->lr_floor >= 0.0f && tp->lr_floor <= 1.0f) || tp->log_every < 0 ||
        (tp->log_every > 0 && !loss_log))
        return set_error(HP_ERR_ARG, "hp_sur_train: bad arguments");
    cudaStream_t s = as_stream(stream);
    // minibatches of whole row groups taken in turn; a batch of 0 (or above M) is every row
    const int64_t groups = M / tp->group;
    int64_t B = tp->batch == 0 ? M : (tp->batch / tp->group) * tp->group;
    if (B > M) B = M;
    if (B < 1 || groups < 1) return set_error(HP_ERR_ARG, "hp_sur_train: batch smaller than one row group");
    const int64_t n_batches = M / B > 0 ? M / B : 1;
    float* lbuf = nullptr;
    if (cudaMallocAsync((void**)&lbuf, sizeof(float), s) != cudaSuccess)
        return set_error(HP_ERR_OOM, "hp_sur_train: allocation failed");
    MlpTrain tr;
    int rc = mlp_train_begin(params, B, &tr, s);
    const double pi = 3.14159265358979323846;
    // per step: cosine decay from lr to lr_floor * lr over the run, and Adam's bias corrections
    std::vector<float> sched(3 * (size_t)(tp->steps > 0 ? tp->steps : 1));
    for (int32_t step = 1; step <= tp->steps; ++step) {
        const double c = 0.5 * (1.0 + cos(pi * (double)step / (double)tp->steps));
        sched[3 * (size_t)(step - 1)] =
            (float)((double)tp->lr * ((double)tp->lr_floor + (1.0 - (double)tp->lr_floor) * c));
        sched[3 * (size_t)(step - 1) + 1] = 1.0f - powf(tp->beta1, (float)(step0 + step));
        sched[3 * (size_t)(step - 1) + 2] = 1.0f - powf(tp->beta2, (float)(step0 + step));
    }
    bool ran = false;
    if (rc == HP_OK && tp->steps > 0) {
        // the whole run as one persistent launch when every CTA can stay resident
        float *dsched = nullptr, *dlog = nullptr;
        cudaError_t e = cudaMallocAsync((void**)&dsched, sizeof(float) * sched.size(), s);
        if (e == cudaSuccess && tp->log_every > 0) e = cudaMallocAsync((void**)&dlog, sizeof(float) * tp->steps, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(dsched, sched.data(), sizeof(float) * sched.size(), cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) rc = cuda_error(e, "hp_sur_train: schedule");
        if (rc == HP_OK)
            rc = mlp_train_loop(&tr, params, m, v, X, Y, n_batches, tp->steps, dsched, tp->beta1, tp->beta2, tp->eps,
                                dlog, lbuf, s, &ran);
        if (rc == HP_OK && ran && tp->log_every > 0) {
            std::vector<float> h((size_t)tp->steps);
            e = cudaMemcpyAsync(h.data(), dlog, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) rc = cuda_error(e, "hp_sur_train: loss read-back");
            for (int32_t k = 0; k < tp->steps / tp->log_every; ++k) loss_log[k] = h[(size_t)(k + 1) * tp->log_every - 1];
        }
        // the schedule's host copy must outlive the upload
        const cudaError_t e2 = cudaStreamSynchronize(s);
        if (e2 != cudaSuccess && rc == HP_OK) rc = cuda_error(e2, "hp_sur_train");
        cudaFreeAsync(dsched, s);
        if (dlog) cudaFreeAsync(dlog, s);
    }
    for (int32_t step = 1; !ran && step <= tp->steps && rc == HP_OK; ++step) {
        const int64_t r0 = ((int64_t)(step - 1) % n_batches) * B;
        rc = mlp_train_step(&tr, params, m, v, X + 11 * r0, Y + 2 * r0, step0 + step, sched[3 * (size_t)(step - 1)],
                            tp->beta1, tp->beta2, tp->eps, lbuf, s);
        if (rc == HP_OK && tp->log_every > 0 && step % tp->log_every == 0) {
            float h = 0.0f;
            cudaError_t e = cudaMemcpyAsync(&h, lbuf, sizeof(float), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) rc = cuda_error(e, "hp_sur_train: loss read-back");
            loss_log[step / tp->log_every - 1] = h;
        }
    }
    if (rc == HP_OK && loss && tp->steps > 0) {
        const cudaError_t e = cudaMemcpyAsync(loss, lbuf, sizeof(float), cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) rc = cuda_error(e, "hp_sur_train: loss copy");
    }
    mlp_train_end(&tr, s);
    cudaFreeAsync(lbuf, s);
    const cudaError_t e = cudaStreamSynchronize(s);  // both paths return with the run finished
    if (e != cudaSuccess && rc == HP_OK) rc = cuda_error(e, "hp_sur_train");
    return rc;
}
