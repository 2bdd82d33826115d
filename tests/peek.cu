// peek.cu -- what the tests read from and set in a handle beyond the C ABI.
#include "ad_internal.cuh"

extern "C" int peek_degrees(ad_graph_t g, double *D, uint8_t *exact) {
    if (cudaStreamSynchronize(g->stream) != cudaSuccess) return 1;
    if (cudaMemcpy(D, g->D, g->n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    return cudaMemcpy(exact, g->dexact, g->n, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 3;
}

extern "C" void peek_set_shape(ad_graph_t g, int32_t R, int32_t storage, int32_t lanes, int32_t chunks) {
    g->tuned.push_back({R, storage, lanes, chunks, 0});
}
