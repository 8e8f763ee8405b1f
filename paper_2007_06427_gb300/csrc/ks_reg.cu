// ks_reg.cu - the instances of the float register kernels (ks_reg.cuh), a translation unit of their own so
// that the library's kernels compile side by side.
#include "ks_reg.cuh"

namespace ks {

template <int MODE>
static RgRowsFn rows_fn(int lgnx) {
    switch (lgnx) {
    case 5: return k_rg_rows<MODE, 5>;
    case 6: return k_rg_rows<MODE, 6>;
    case 7: return k_rg_rows<MODE, 7>;
    case 8: return k_rg_rows<MODE, 8>;
    default: return k_rg_rows<MODE, 9>;
    }
}
RgRowsFn rg_rows_fn(int mode, int lgnx) { return mode == ROW_NONLIN ? rows_fn<ROW_NONLIN>(lgnx) : rows_fn<ROW_ADJ>(lgnx); }
RgColsFn rg_cols_fn(int mode) { return mode == COL_RESID ? k_rg_cols<COL_RESID> : k_rg_cols<COL_UPDATE>; }

}  // namespace ks
