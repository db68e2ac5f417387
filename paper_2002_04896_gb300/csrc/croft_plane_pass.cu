// croft_plane_pass.cu - the z+y pass over whole yz-planes (croft_plane_pass_kernel.cuh): kernel
// lookup, tables and launch.
#include "croft_plane_pass_kernel.cuh"

namespace croft {

plane_pass_fn plane_pass_kernel_for(int ny) {
    switch (ny) {
#define CROFT_PLANE_Y(NY) \
    case NY: return croft_plane_pass_kernel<NY>;
        CROFT_PLANE_Y_SIZES(CROFT_PLANE_Y)
#undef CROFT_PLANE_Y
        default: return nullptr;
    }
}

cudaError_t plane_pass_prepare(int ny, int smem) {
    plane_pass_fn f = plane_pass_kernel_for(ny);
    if (!f) return cudaErrorInvalidValue;
    return allow_smem((const void*)f, smem);
}

cudaError_t launch_plane_pass(const PlanePass& P, const float2* in, float2* out, float isign, cudaStream_t s, bool pdl) {
    PlanePassArgs A = P.args;
    A.in = in;
    A.out = out;
    A.isign = isign;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P.grid, 1, 1);
    cfg.blockDim = dim3((unsigned)P.block, 1, 1);
    cfg.dynamicSmemBytes = (size_t)P.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (pdl) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, P.fn, A);
}

}  // namespace croft
