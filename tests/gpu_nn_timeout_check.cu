// A training step whose device-side wait gave up (the error word set here, as the kernels set it): the parameters and Adam
// moments stay, the next call that synchronises reports it once, and training goes on afterwards. Exit status 0 on success.
#include "nn.cu"

#include <cstdio>

static int run(int n) {
    const size_t nv = (size_t)n * n * n;
    std::vector<float> h(3 * nv);
    for (size_t i = 0; i < h.size(); ++i) h[i] = (float)((i * 2654435761u >> 8) % 1000) * 0.001f - 0.5f;
    float *psi = nullptr, *tgt = nullptr;
    if (cudaMalloc(&psi, h.size() * 4) || cudaMalloc(&tgt, h.size() * 4)) return 1;
    cudaMemcpy(psi, h.data(), h.size() * 4, cudaMemcpyHostToDevice);
    for (auto& v : h) v = 0.3f * v * v;
    cudaMemcpy(tgt, h.data(), h.size() * 4, cudaMemcpyHostToDevice);
    colapm_nn_config cfg;
    colapm_nn_default_config(&cfg);
    colapm_nn* c = nullptr;
    if (colapm_nn_create(n, &cfg, nullptr, &c)) return 2;
    std::vector<float> p0(COLAPM_NN_PARAMS), p1(p0), m0((size_t)LAYERS * LSIZE), m1(m0);
    double loss = 0.0;
    int bad = 0;
    auto expect = [&](const char* what, bool ok) {
        if (!ok) std::printf("n=%d: %s\n", n, what);
        bad |= !ok;
    };
    auto moments = [&](std::vector<float>& m) { return cudaMemcpy(m.data(), c->m1, m.size() * 4, cudaMemcpyDeviceToHost); };
    const int four = 4;
    auto give_up = [&] { return cudaMemcpy(c->err, &four, sizeof(four), cudaMemcpyHostToDevice); };
    expect("first step", !colapm_nn_train_step(c, psi, tgt, &loss) && !colapm_nn_get_params(c, p0.data()) && !moments(m0));
    give_up();
    expect("a step without a loss does not wait", !colapm_nn_train_step(c, psi, tgt, nullptr));
    expect("reading the parameters reports the timeout", colapm_nn_get_params(c, p1.data()) == COLAPM_E_TIMEOUT);
    expect("and only once", colapm_nn_get_params(c, p1.data()) == COLAPM_OK);
    expect("the parameters stay", p0 == p1);
    moments(m1);
    expect("the moments stay", m0 == m1);
    give_up();
    expect("a step with a loss reports it", colapm_nn_train_step(c, psi, tgt, &loss) == COLAPM_E_TIMEOUT);
    expect("and leaves the parameters", !colapm_nn_get_params(c, p1.data()) && p0 == p1);
    expect("training goes on", !colapm_nn_train_step(c, psi, tgt, &loss) && !colapm_nn_get_params(c, p1.data()) && p0 != p1);
    colapm_nn_destroy(c);
    cudaFree(psi);
    cudaFree(tgt);
    return bad;
}

int main() { return run(16) | run(48); }
