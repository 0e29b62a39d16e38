// itc_fields_tma.cu -- the tensor-tile fields kernel (itc_fields_tma.cuh) for absolute moments and for 32-
// and 128-row tiles, radii 6, 9 and 12, and the dispatch over every compiled form.
#include "itc_fields_tma.cuh"

namespace itc {
namespace {

template <bool ABS, int DTYPE, int TH>
cudaError_t dispatch(const FieldsLaunch& L, int ntiles, int R, cudaStream_t s) {
    if (R == 6) return launch_tma<6, ABS, DTYPE, TH, false>(L, ntiles, s);
    if (R == 9) return launch_tma<9, ABS, DTYPE, TH, false>(L, ntiles, s);
    if (R == 12) return launch_tma<12, ABS, DTYPE, TH, false>(L, ntiles, s);
    return cudaErrorInvalidValue;
}

template <int DTYPE>
cudaError_t dispatch_height(const FieldsLaunch& L, int ntiles, int R, cudaStream_t s) {
    if (L.absolute)
        return L.tile_h == 128  ? dispatch<true, DTYPE, 128>(L, ntiles, R, s)
               : L.tile_h == 32 ? dispatch<true, DTYPE, 32>(L, ntiles, R, s)
                                : dispatch<true, DTYPE, 64>(L, ntiles, R, s);
    return L.tile_h == 128 ? dispatch<false, DTYPE, 128>(L, ntiles, R, s) : dispatch<false, DTYPE, 32>(L, ntiles, R, s);
}

}  // namespace

bool fields_stg_supported(int ndim, int dtype, int Ru, int Rv, bool absolute) {
    return !absolute && fields_tma_supported(ndim, dtype, Ru, Rv, false);
}

cudaError_t launch_fields_stg(const FieldsLaunch& L, int ntiles, int R, int dtype, cudaStream_t s) {
    if (ntiles - L.tile_base <= 0) return cudaSuccess;
    if (!L.counter || L.absolute) return cudaErrorInvalidValue;
    if (L.mode) return dtype == ITC_U8 ? launch_fields_stg_self_u8(L, ntiles, R, s) : launch_fields_stg_self_f32(L, ntiles, R, s);
    return dtype == ITC_U8 ? launch_fields_stg_u8(L, ntiles, R, s) : launch_fields_stg_f32(L, ntiles, R, s);
}

bool fields_tma_heights(int R) { return R == 6 || R == 9 || R == 12; }

bool fields_tma_supported(int ndim, int dtype, int Ru, int Rv, bool absolute) {
    if (ndim != 2 || Ru != Rv) return false;
    return absolute ? fields_tma_heights(Ru) : Ru >= 3 && Ru <= (dtype == ITC_U8 ? 16 : 12);
}

int fields_tma_box(int dtype, int R, int tile_h, int* box_w, int* box_h) {
    const int ra = dtype == ITC_U8 ? 16 : ((R + 3) & ~3);
    *box_w = kTileW + 2 * ra;
    *box_h = tile_h + 2 * R;
    return 0;
}

cudaError_t launch_fields_tma(const FieldsLaunch& L, int ntiles, int R, int dtype, cudaStream_t s) {
    if (ntiles - L.tile_base <= 0) return cudaSuccess;
    if (!L.counter) return cudaErrorInvalidValue;   // the tile counter is required (zeroed by the caller)
    if (L.mode) return dtype == ITC_U8 ? launch_fields_tma_self_u8(L, ntiles, R, s) : launch_fields_tma_self_f32(L, ntiles, R, s);
    if (!L.absolute && L.tile_h == 64)
        return dtype == ITC_U8 ? launch_fields_tma_u8(L, ntiles, R, s) : launch_fields_tma_f32(L, ntiles, R, s);
    return dtype == ITC_U8 ? dispatch_height<ITC_U8>(L, ntiles, R, s) : dispatch_height<ITC_F32>(L, ntiles, R, s);
}

}  // namespace itc
