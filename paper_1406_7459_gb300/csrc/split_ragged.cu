// split_ragged.cu -- the split pass 2 of ragged thick samples: y lines of the
// carrier lengths of ragged.cuh, z columns of 1, 2, 4, 8 (one y position per
// thread) or 16 ... 128 with the lengths between the powers of two.  They
// replace the mixed-radix kernels (split_kernels.cu) wherever a carrier
// length exists; those remain for sides above 1024 and more than 128 layers.
// Per launch on 100x80x20, general kernels against these: y transforms 12.7
// against 7.6 us, z with the product 35 against 14.6, update 16.9 against
// 12.1; ten steps and the energy 833 against 547 us.  Bound by the shared-
// memory round trips and barriers of short lines.
#include "ragged.cuh"
#include "split_fast.cuh"

namespace mmk {

template <int NY> static bool fill_y(FastSplitFns* f) {
    f->yf = k_yfwd_fast<NY, true>;
    f->yi = k_yinv_fast<NY, true>;
    f->ylpc = YLayout<NY>::LPC;
    f->ty = YLayout<NY>::THREADS;
    f->sy = YLayout<NY>::RAG_BYTES;
    return true;
}
template <int NZ> static int fill_z(FastSplitFns* f) {
    f->zc = k_zconv_fast<NZ, true>;
    f->zw = ZLayout<NZ>::W;
    f->tz = ZLayout<NZ>::THREADS;
    f->sz = ZLayout<NZ>::BYTES;
    return NZ;
}
template <int NZ> static int fill_zcol(FastSplitFns* f) {
    f->zc = k_zcol_fast<NZ, true>;
    f->zw = 0;                               // marks the one-position-per-thread kernel
    f->tz = kZcolThreads;
    f->sz = 0;
    return NZ;
}

bool ragged_split_lookup(int ny, int nz, FastSplitFns* f, int* NY, int* NZ) {
    *NY = ragged_len(ny);
    bool ok = false;
    switch (*NY) {
        case 16: ok = fill_y<16>(f); break;
        case 32: ok = fill_y<32>(f); break;
        case 48: ok = fill_y<48>(f); break;
        case 64: ok = fill_y<64>(f); break;
        case 96: ok = fill_y<96>(f); break;
        case 128: ok = fill_y<128>(f); break;
        case 192: ok = fill_y<192>(f); break;
        case 256: ok = fill_y<256>(f); break;
        case 320: ok = fill_y<320>(f); break;
        case 384: ok = fill_y<384>(f); break;
        case 512: ok = fill_y<512>(f); break;
        case 640: ok = fill_y<640>(f); break;
        case 768: ok = fill_y<768>(f); break;
        case 1024: ok = fill_y<1024>(f); break;
        default: break;
    }
    if (!ok) return false;
    *NZ = nz <= 1     ? fill_zcol<1>(f)
          : nz <= 2   ? fill_zcol<2>(f)
          : nz <= 4   ? fill_zcol<4>(f)
          : nz <= 8   ? fill_zcol<8>(f)
          : nz <= 16  ? fill_z<16>(f)
          : nz <= 24  ? fill_z<24>(f)
          : nz <= 32  ? fill_z<32>(f)
          : nz <= 48  ? fill_z<48>(f)
          : nz <= 64  ? fill_z<64>(f)
          : nz <= 96  ? fill_z<96>(f)
          : nz <= 128 ? fill_z<128>(f)
                      : 0;
    return *NZ != 0;
}

}  // namespace mmk
