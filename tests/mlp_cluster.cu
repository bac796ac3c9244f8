// The training and gradient kernels with the cluster size given by the test:
// the library takes 16 blocks and falls back to 8 where the device has no room
// for 16.  Compiled by test_gpu_mlp_cluster.py against the built library.
#include "../paper_0909_0541_gb300/csrc/nb_mlp.cu"

template <bool TRAIN>
static int run(int blocks, float *P, float *m, float *v, const float *feat, const float *labels,
               const int32_t *order, int64_t n, int64_t batch, int64_t total, float lr, float *grad,
               float *loss, void *work, cudaStream_t s)
{
    TrainShare *share = (TrainShare *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
    const int64_t spe = n / batch;
    for (int64_t k = 0; k < total; k += MT_STEPS) {
        const int steps = (int)(total - k < MT_STEPS ? total - k : MT_STEPS);
        bool runs = false;
        const cudaError_t e =
            blocks == 16 ? launch_train_cl<16, TRAIN>(P, m, v, feat, labels, order, n, batch, spe,
                                                      k, steps, lr, share, grad, loss, s, &runs)
                         : launch_train_cl<8, TRAIN>(P, m, v, feat, labels, order, n, batch, spe, k,
                                                     steps, lr, share, grad, loss, s, &runs);
        if (e != cudaSuccess || !runs) return -1;
    }
    return 0;
}

extern "C" int cluster_train(int blocks, float *P, float *m, float *v, const float *feat,
                             const float *labels, const int32_t *order, int64_t n, int epochs,
                             int64_t batch, float lr, float *loss, void *work, void *stream)
{
    return run<true>(blocks, P, m, v, feat, labels, order, n, batch, (n / batch) * epochs, lr,
                     nullptr, loss, work, (cudaStream_t)stream);
}

extern "C" int cluster_grad(int blocks, const float *P, const float *feat, const float *labels,
                            int64_t n, float *grad, float *loss, void *work, void *stream)
{
    return run<false>(blocks, const_cast<float *>(P), nullptr, nullptr, feat, labels, nullptr, n, n,
                      1, 0.f, grad, loss, work, (cudaStream_t)stream);
}
