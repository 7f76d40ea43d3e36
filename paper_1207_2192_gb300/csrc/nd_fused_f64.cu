// nd_fused_f64.cu -- instantiations of the fused on-chip kernel in FP64.
#include "nd_field_impl.cuh"

namespace nd {

size_t fused_smem_f64(int P, int D, int Dpad, bool wbuf, int variant)
{
    const int nt = fused_nt(P, variant);
    if (nt == 0) return (size_t)-1;
    switch (P) {
    case 16: return fused_smem_bytes<16, double>(D, Dpad, nt, wbuf);
    case 32: return fused_smem_bytes<32, double>(D, Dpad, nt, wbuf);
    case 64: return fused_smem_bytes<64, double>(D, Dpad, nt, wbuf);
    default: return (size_t)-1;
    }
}

template <int P>
static int occ_p(int mode, size_t smem, int variant)
{
    switch (mode) {
    case M_RK4: return fused_occupancy<P, double, M_RK4>(variant, smem);
    case M_HEUN: return fused_occupancy<P, double, M_HEUN>(variant, smem);
    default: return 0;
    }
}

int fused_blocks_per_sm_f64(int P, int mode, size_t smem, int variant)
{
    switch (P) {
    case 16: return occ_p<16>(mode, smem, variant);
    case 32: return occ_p<32>(mode, smem, variant);
    case 64: return occ_p<64>(mode, smem, variant);
    default: return 0;
    }
}

int fused_variant_threads_f64(int P, int variant) { return fused_nt(P, variant); }

cudaError_t launch_fused_f64(int P, const LaunchArgs &a)
{
    switch (P) {
    case 16: return launch_fused_p<16, double>(a);
    case 32: return launch_fused_p<32, double>(a);
    case 64: return launch_fused_p<64, double>(a);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace nd
