// One checkpoint saved and restored by the library's own functions, which are
// internal to their source file.
#include "mmod_adjoint.cu"

extern "C" __attribute__((visibility("default"))) int roundtrip(int dtype, int nxp, int ny, int nz, float *u_prev,
                                                                float *u_cur, float *v_prev, float *v_cur, void *stored,
                                                                float *scales, void *stream) {
    mmod_handle h;
    h.cfg.nz = nz;
    h.nxp = nxp;
    h.plane = (long long)nxp * ny;
    h.vol = h.plane * nz;
    h.gw.dtype = dtype;
    h.gw.ckpt = stored;
    h.gw.ckpt_scale = scales;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaError_t e = save_state(&h, 0, u_prev, u_cur, s)) return (int)e;
    return (int)restore_state(&h, 0, v_prev, v_cur, s);
}
