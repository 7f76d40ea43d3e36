// nd_fused_f32.cu -- instantiations of the fused on-chip kernel in FP32.
#include "nd_field_impl.cuh"

namespace nd {

size_t fused_smem_f32(int P, int D, int Dpad, bool wbuf, int variant)
{
    const int nt = fused_nt(P, variant);
    if (nt == 0) return (size_t)-1;
    switch (P) {
    case 16: return fused_smem_bytes<16, float>(D, Dpad, nt, wbuf);
    case 32: return fused_smem_bytes<32, float>(D, Dpad, nt, wbuf);
    case 64: return fused_smem_bytes<64, float>(D, Dpad, nt, wbuf);
    case 128: return fused_smem_bytes<128, float>(D, Dpad, nt, wbuf);
    default: return (size_t)-1;
    }
}

template <int P>
static int occ_p(int mode, size_t smem, int variant)
{
    switch (mode) {
    case M_RK4: return fused_occupancy<P, float, M_RK4>(variant, smem);
    case M_HEUN: return fused_occupancy<P, float, M_HEUN>(variant, smem);
    default: return 0;
    }
}

int fused_blocks_per_sm_f32(int P, int mode, size_t smem, int variant)
{
    switch (P) {
    case 16: return occ_p<16>(mode, smem, variant);
    case 32: return occ_p<32>(mode, smem, variant);
    case 64: return occ_p<64>(mode, smem, variant);
    case 128: return occ_p<128>(mode, smem, variant);
    default: return 0;
    }
}

int fused_variant_threads_f32(int P, int variant) { return fused_nt(P, variant); }

cudaError_t launch_fused_f32(int P, const LaunchArgs &a)
{
    switch (P) {
    case 16: return launch_fused_p<16, float>(a);
    case 32: return launch_fused_p<32, float>(a);
    case 64: return launch_fused_p<64, float>(a);
    case 128: return launch_fused_p<128, float>(a);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace nd
