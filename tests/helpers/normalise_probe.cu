// Device-side normalisation of n-vectors (nvec.cuh) beside the plain quotient
// by the root, for the test that compares their bits.
#include "nvec.cuh"

using namespace pyro;

template <int NC, typename T>
__global__ void probe(const T *in, T *fast, T *plain, long n)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    using A = Ar<T>;
    T t[NC];
    for (int k = 0; k < NC; ++k) t[k] = in[NC * i + k];
    T q = A::mul(t[0], t[0]);
    for (int k = 1; k < NC; ++k) q = A::add(q, A::mul(t[k], t[k]));
    q = A::sqrt_(q);
    for (int k = 0; k < NC; ++k) plain[NC * i + k] = A::div(t[k], q);
    normalise<NC>(t);
    for (int k = 0; k < NC; ++k) fast[NC * i + k] = t[k];
}

template <int NC, typename T>
static int run(const void *in, void *fast, void *plain, long n)
{
    probe<NC, T><<<(unsigned)((n + 255) / 256), 256>>>((const T *)in, (T *)fast, (T *)plain, n);
    return (int)cudaDeviceSynchronize();
}

// n vectors of nc components, device arrays of float (bits = 32) or double.
extern "C" int probe_normalise(int nc, int bits, const void *in, void *fast, void *plain, long n)
{
    if (nc == 2) return bits == 32 ? run<2, float>(in, fast, plain, n) : run<2, double>(in, fast, plain, n);
    return bits == 32 ? run<3, float>(in, fast, plain, n) : run<3, double>(in, fast, plain, n);
}
