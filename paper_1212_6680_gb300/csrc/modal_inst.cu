// modal_inst.cu -- one lane configuration of the mode-space kernels (compiled once per
// (SMG_MG, SMG_MK, SMG_MT): G lanes a plane, K lines a lane, MT 0 float, 1 double).
#include "modal.cuh"

namespace smg {
namespace {

constexpr int G = SMG_MG, K = SMG_MK;
#if SMG_MT == 0
using T = float;
#else
using T = double;
#endif

cudaError_t setup(const ModalArgs<T> &a, T *coef, double *coef64, cudaStream_t st) {
    const long long jobs = static_cast<long long>(a.nmode) * a.ncls_all;
    const size_t smem = sizeof(double) * 4 * a.ntype * kRow;
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&modal_setup_kernel<T, G, K>), smem);
    if (e != cudaSuccess) return e;
    modal_setup_kernel<T, G, K><<<static_cast<unsigned>((jobs + 3) / 4), 128, smem, st>>>(a, coef, coef64);
    return cudaGetLastError();
}

cudaError_t tail(const ModalArgs<T> *d_args, int nmode, int nb, int coarse_iters, int threads, size_t smem, cudaStream_t st) {
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&modal_tail_kernel<T, G, K>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(modal_tail_kernel<T, G, K>, dim3(nmode, nb), dim3(threads), smem, st, d_args, coarse_iters);
}

cudaError_t tail_batch(const ModalArgs<T> *d_args, const ModalTask *tasks, int ntasks, const int *active, int threads, size_t smem,
                       cudaStream_t st) {
#if SMG_MT == 0
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&modal_tail_batch_kernel<T, G, K>), smem);
    if (e != cudaSuccess) return e;
    modal_tail_batch_kernel<T, G, K><<<ntasks, threads, smem, st>>>(d_args, tasks, active);
    return cudaGetLastError();
#else
    return cudaErrorNotSupported;  // the batched solver runs FP32 cycles
#endif
}

// The slab's coarse planes: as many as its red planes (the slab's share + 3) fit in one pass over the
// groups, in at most half of an SM's shared memory (two CTAs per SM) where that holds a useful slab: four coarse planes,
// 13 rows (256^3 and 384^3 with two coarse planes, or one CTA an SM always: within 1 %).
int slab_count(const ModalArgs<T> &a, int l, size_t *smem) {
    const int groups = modal_threads<T>() / G, nzc = a.nz[l + 1];
    const size_t row = static_cast<size_t>(a.sm_pitch) * sizeof(T), tabs = static_cast<size_t>(a.ncls[l]) * Tab<G, K>::kElems * sizeof(T);
    const size_t half = kModalSmem / 2;
    long long rows = tabs + 13 * row <= half ? static_cast<long long>((half - tabs) / row)
                                             : static_cast<long long>((kModalSmem - std::min(kModalSmem, tabs)) / row);
    const int most = static_cast<int>(std::min<long long>(groups - 3, (rows - 5) / 2));
    if (most < 1) return 0;
    const int n = (nzc + most - 1) / most, z = (nzc + n - 1) / n;
    if (smem) *smem = tabs + static_cast<size_t>(2 * z + 5) * row;
    return n;
}

bool slab_fits(const ModalArgs<T> &a, int l) { return slab_count(a, l, nullptr) > 0; }

cudaError_t slab(const ModalArgs<T> &a, int l, int nb, cudaStream_t st) {
    size_t smem = 0;
    const int n = slab_count(a, l, &smem);
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&modal_slab_kernel<T, G, K>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(modal_slab_kernel<T, G, K>, dim3(n, a.nmode, nb), dim3(modal_threads<T>()), smem, st, a, l, n);
}

int shares(int planes) { return (planes + 4 * (256 / G) - 1) / (4 * (256 / G)); }  // up to four passes over the groups

cudaError_t relax(const ModalArgs<T> &a, int l, int colour, int mode, int nb, cudaStream_t st) {
    const int n = colour ? a.nz[l] / 2 : (a.nz[l] + 1) / 2;
    if (n == 0) return cudaSuccess;
    const size_t smem = static_cast<size_t>(a.ncls[l]) * Tab<G, K>::kElems * sizeof(T);
    cudaError_t e = raise_smem_attr(reinterpret_cast<const void *>(&modal_relax_kernel<T, G, K>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(modal_relax_kernel<T, G, K>, dim3(shares(n), a.nmode, nb), dim3(256), smem, st, a, l, colour, mode);
}

cudaError_t restrict_(const ModalArgs<T> &a, int l, int nb, cudaStream_t st) {
    return launch_pdl(modal_restrict_kernel<T, G, K>, dim3(shares(a.nz[l + 1]), a.nmode, nb), dim3(256), 0, st, a, l);
}

}  // namespace

#define SMG_CAT_(a, b, c, d) a##b##_##c##_##d
#define SMG_CAT(a, b, c, d) SMG_CAT_(a, b, c, d)
extern const ModalKernels<T> SMG_CAT(modal_kernels_, SMG_MT, SMG_MG, SMG_MK);
const ModalKernels<T> SMG_CAT(modal_kernels_, SMG_MT, SMG_MG, SMG_MK) = {
    setup, tail, tail_batch, slab, relax, restrict_, slab_fits, Tab<G, K>::kElems, modal_threads<T>()};

}  // namespace smg
