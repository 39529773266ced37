// Row-streaming step kernels for R in {2, 4, 6, 8, 12, 16}.
#include "rows_step.cuh"

namespace mfmc {

const RowsLauncher *rows_launcher(int R) {
    static const RowsLauncher w2 = make_rows_launcher<2>();
    static const RowsLauncher w4 = make_rows_launcher<4>();
    static const RowsLauncher w6 = make_rows_launcher<6>();
    static const RowsLauncher w8 = make_rows_launcher<8>();
    static const RowsLauncher w12 = make_rows_launcher<12>();
    static const RowsLauncher w16 = make_rows_launcher<16>();
    switch (R) {
        case 2: return &w2;
        case 4: return &w4;
        case 6: return &w6;
        case 8: return &w8;
        case 12: return &w12;
        case 16: return &w16;
        default: return nullptr;
    }
}

}  // namespace mfmc
