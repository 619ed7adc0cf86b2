// A training step of which a pass has given up a wait (the passes' flag raised by
// hand: the state that k_forward and the others leave then) changes neither the
// parameters nor the step count, is reported once, and training goes on from the
// last applied step as if it had not been. Prints "ok" or the first difference.
#include <cstdio>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/mlp_kernels.cu"

static std::string g_error;
void lskum::set_last_error(const std::string& m) { g_error = m; }

static int bad(const char* what) {
    std::printf("%s (%s)\n", what, g_error.c_str());
    return 1;
}

static void raise_flag(lskum_mlp* h, int passes) {
    cudaMemcpy(h->err.dev, &passes, sizeof(int), cudaMemcpyHostToDevice);
    *h->err.host = 1;
}

int main() {
    const int n = 300;
    std::mt19937 rng(3);
    std::normal_distribution<float> N(0.f, 0.1f);
    float proj[16];
    for (float& x : proj) x = N(rng);
    const int64_t np = lskum_mlp_num_params();
    std::vector<float> p(np), feat(n * 32, 0.f), target(n * 4), a(np), b(np), c(np);
    for (float& x : p) x = N(rng);
    for (int i = 0; i < n; ++i)
        for (int k = 0; k < 21; ++k) feat[i * 32 + k] = 10 * N(rng);
    for (float& x : target) x = N(rng);
    float *fd, *td;
    cudaMalloc(&fd, feat.size() * 4);
    cudaMalloc(&td, target.size() * 4);
    cudaMemcpy(fd, feat.data(), feat.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(td, target.data(), target.size() * 4, cudaMemcpyHostToDevice);
    lskum_mlp *x = nullptr, *y = nullptr;
    if (lskum_mlp_create(512, proj, &x) || lskum_mlp_create(512, proj, &y)) return bad("create");
    double loss = 0.0;
    for (lskum_mlp* h : {x, y})
        if (lskum_mlp_set_params(h, p.data(), np) || lskum_mlp_train_step(h, fd, td, n, 1e-3f, &loss))
            return bad("first step");
    lskum_mlp_get_params(x, a.data(), np);
    if (a == p) return bad("the first step changed nothing");

    // a synchronising step, then two queued ones of which the first fails
    raise_flag(x, kPassForward | kPassWeightGrads);
    if (lskum_mlp_train_step(x, fd, td, n, 1e-3f, &loss) != LSKUM_ERR_TIMEOUT) return bad("step not reported");
    if (g_error != "forward pass, weight gradients: a wait ran out") return bad("passes not named");
    raise_flag(x, kPassBackward);
    if (lskum_mlp_train_step(x, fd, td, n, 1e-3f, nullptr) || lskum_mlp_train_step(x, fd, td, n, 1e-3f, nullptr))
        return bad("queued step");
    if (lskum_mlp_sync(x) != LSKUM_ERR_TIMEOUT) return bad("queued step not reported");
    lskum_mlp_get_params(x, b.data(), np);
    if (b != a) return bad("parameters changed");
    if (lskum_mlp_sync(x)) return bad("reported twice");

    for (lskum_mlp* h : {x, y})
        if (lskum_mlp_train_step(h, fd, td, n, 1e-3f, &loss)) return bad("second step");
    lskum_mlp_get_params(x, b.data(), np);
    lskum_mlp_get_params(y, c.data(), np);
    if (b == a || b != c) return bad("training did not go on from the last applied step");

    // new parameters clear a failure
    raise_flag(x, kPassForward);
    if (lskum_mlp_set_params(x, p.data(), np) || lskum_mlp_train_step(x, fd, td, n, 1e-3f, &loss))
        return bad("after set_params");
    lskum_mlp_get_params(x, b.data(), np);
    if (b != a) return bad("first step again");
    lskum_mlp_destroy(x);
    lskum_mlp_destroy(y);
    if (cudaDeviceSynchronize() != cudaSuccess) return bad("CUDA");
    std::printf("ok\n");
    return 0;
}
