// The stride-scan and read kernel instances <512, 1>: 512-thread blocks, or grids of at
// most two blocks per SM.
#include "gfs_scan.cuh"

namespace gfs {

cudaError_t launch_scan_wide(const DevHandle& g, int fid, const gfs_scan_args& a, unsigned long long nstrides,
                        int64_t* d_count, uint64_t* d_sum, uint64_t* d_hash, cudaStream_t s) {
  return launch_scan_as<512, 1>(g, fid, a, nstrides, d_count, d_sum, d_hash, s);
}

cudaError_t scan_setup_wide() { return scan_setup_as<512, 1>(); }

cudaError_t scan_occupancy_wide(int threads, int* per_sm) { return scan_occupancy_as<512, 1>(threads, per_sm); }

void launch_read_many_wide(const DevHandle& g, int fid, uint32_t n, const uint64_t* d_off, const uint64_t* d_len,
                      const uint64_t* d_dst, uint8_t* d_buf, int64_t* d_ret, uint32_t blocks, uint32_t threads,
                      bool cold, cudaStream_t s) {
  const dev::ReadList list{d_off, d_len, d_dst, d_buf, (long long*)d_ret, n};
  if (cold) k_read_many<false, 512, 1><<<blocks, threads, 0, s>>>(g, fid, list);
  else k_read_many<true, 512, 1><<<blocks, threads, 0, s>>>(g, fid, list);
}

}  // namespace gfs
