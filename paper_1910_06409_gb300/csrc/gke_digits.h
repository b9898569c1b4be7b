// gke_digits.h -- FP64 contractions over snapshots from exact digit products on
// the tensor cores (internal; gke_digits.cu describes the method).
#pragma once
#include <cuda_runtime.h>
#include <string>
#include "../../include/gke.h"
#include "gke_common.cuh"

namespace gke {

struct DigitWork {
    void* ws = nullptr;         // digit operands and row exponents of one chunk of wavenumbers
    size_t bytes = 0;
    int* err = nullptr;         // device flag: a pipeline wait timed out
};

// operands are made and used in chunks of wavenumbers of this many bytes at most
constexpr size_t DG_CHUNK_BYTES = (size_t)512 << 20;
// workspace for chunks of up to Kc wavenumbers of `per` bytes each, `limit`
// bytes (but one wavenumber) at most; where the device has less free, half of it
// and so on.  Only where one wavenumber's operands find no room the work stays
// empty (digits_ready false) and the callers keep their FMA kernels;
// st: the stream of the passes (the error flag is cleared in its order)
void digits_alloc(DigitWork& w, size_t per, int Kc, cudaStream_t st, size_t limit = DG_CHUNK_BYTES);
inline bool digits_ready(const DigitWork& w) { return w.ws != nullptr; }
// the channel's kernels and workspace (n wall-normal points)
cudaError_t digits_setup(DigitWork& w, int n, int Kc, cudaStream_t st);
size_t digits_per_k(int n);                 // bytes of one wavenumber
// whether the digit products are the faster way for a batch (measured; gke_digits.cu)
bool digits_pays(int n, int ns, long long Kc);
// the contractions `jobs` of the wavenumbers [k0, k0 + Kc) into raw (as
// correlate_launch's FP64 form); *launches gets the kernels launched
gke_status digits_correlate(DigitWork& w, const zd* Xop, int ns, int ny, int Nk, int k0, int Kc, zd* raw,
                            unsigned jobs, cudaStream_t st, std::string& err, int* launches);
gke_status digits_check(DigitWork& w, cudaStream_t st, std::string& err);
void digits_free(DigitWork& w);

}  // namespace gke
