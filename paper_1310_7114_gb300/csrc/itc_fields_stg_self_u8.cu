// itc_fields_stg_self_u8.cu -- the tiled fields kernel (itc_fields_tma.cuh): bytes, the self-overlap pass, rows on any boundary.
#include "itc_fields_tma.cuh"

namespace itc {

cudaError_t launch_fields_stg_self_u8(const FieldsLaunch& L, int ntiles, int R, cudaStream_t s) {
    switch (R) {
        case 3: return launch_tma<3, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 4: return launch_tma<4, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 5: return launch_tma<5, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 6: return launch_tma<6, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 7: return launch_tma<7, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 8: return launch_tma<8, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 9: return launch_tma<9, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 10: return launch_tma<10, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 11: return launch_tma<11, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 12: return launch_tma<12, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 13: return launch_tma<13, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 14: return launch_tma<14, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 15: return launch_tma<15, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        case 16: return launch_tma<16, false, ITC_U8, 64, true, true, kAny>(L, ntiles, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace itc
