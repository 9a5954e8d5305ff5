// k_step_f32.cu -- stencil and persistent kernels for f32 vector storage.
#include "k_stencil.cuh"
#include "k_rows.cuh"
#include "k_col.cuh"

namespace tls {

cudaError_t launch_step_f32(const StepArgs &a) { return step_dispatch<P_F32>(a); }
cudaError_t launch_step_il_f32(const StepArgs &a) { return step_il_dispatch<P_F32>(a); }
cudaError_t launch_step_col_f32(const StepArgs &a) { return col_dispatch<P_F32>(a); }
cudaError_t launch_step_zm_f32(const StepArgs &a) { return step_zm_dispatch<P_F32>(a); }
cudaError_t launch_step_rows_f32(const StepArgs &a, int *err) { return rows_dispatch<P_F32>(a, err); }
cudaError_t launch_persistent_f32(const PersistArgs &a) { return persist_dispatch<P_F32>(a); }
int persistent_occupancy_f32(int wfmt, int vb, int threads) { return occ_dispatch<P_F32>(wfmt, vb, threads); }

bool col_map(CUtensorMap &m, const char *W, const SubGeom &g, int nblk, int wb, int sites)
{
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                               const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<Encode>(f);
    }();
    if (!encode || sites < 1 || 2 * sites > 256) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)(2 * g.Ps), (cuuint64_t)(wb / 16), (cuuint64_t)(3 * (int64_t)nblk)};
    const cuuint64_t strides[2] = {(cuuint64_t)(16 * g.Ps), (cuuint64_t)((int64_t)wb * g.Ps)};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * sites), (cuuint32_t)(wb / 16), 1}, step[3] = {1, 1, 1};
    return encode(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<char *>(W), dims, strides, box, step,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool rows_applicable(int wfmt, int prec, const SubGeom &g, int nvec, int vb, int max_smem)
{
    if (prec == P_F64) return false;
    return rows_ok(wfmt, prec, g, nvec, vb, max_smem);
}

}  // namespace tls
