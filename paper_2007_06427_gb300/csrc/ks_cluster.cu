// ks_cluster.cu - the instances of the cluster kernel (ks_cluster.cuh), a translation unit of their own so
// that the library's kernels compile side by side.
#include "ks_cluster.cuh"

namespace ks {

template <typename R, typename RA>
ClusterFn<R, RA> cluster_fn(bool xi, int mb) {
    if (mb == 2) return xi ? k_cluster<R, RA, true, 2> : k_cluster<R, RA, false, 2>;
    return xi ? k_cluster<R, RA, true, 1> : k_cluster<R, RA, false, 1>;
}
template ClusterFn<double, double> cluster_fn<double, double>(bool, int);
template ClusterFn<float, float> cluster_fn<float, float>(bool, int);
template ClusterFn<double, float> cluster_fn<double, float>(bool, int);

}  // namespace ks
