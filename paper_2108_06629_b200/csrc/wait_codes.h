// Status words of bounded waits that expired: which role of which kernel gave up.  No value is used twice, and a
// status word keeps the first one written to it, so the word names the wait that failed and not one that failed
// in its wake.  Shared by the kernels and the host's messages.
#pragma once

namespace lp {

enum WaitCode {
  WAIT_GEMM_PRODUCER = 1, WAIT_GEMM_MMA = 2, WAIT_GEMM_EPILOGUE = 3, WAIT_GEMM_CHUNK = 4,                        // gemm.cuh
  WAIT_CLUSTER_PRODUCER = 5, WAIT_CLUSTER_MMA = 6, WAIT_CLUSTER_EPILOGUE = 7,                                    // gemmc.cuh
  WAIT_HALO_PRODUCER = 8, WAIT_HALO_MMA = 9, WAIT_HALO_EPILOGUE = 10,                                            // conv_halo.cuh
  WAIT_PAIR_PRODUCER = 11, WAIT_PAIR_MMA = 12, WAIT_PAIR_EPILOGUE = 13, WAIT_PAIR_CHUNK = 14,                    // gemm2.cuh
  WAIT_PAIR_G_PRODUCER = 15, WAIT_PAIR_G_MMA = 16, WAIT_PAIR_G_UPDATE_PRODUCER = 17, WAIT_PAIR_G_EPILOGUE = 18,  // gemm2p.cuh
  WAIT_PAIR_G_CHUNK = 19,
  WAIT_HALO_G_PRODUCER = 21, WAIT_HALO_G_MMA = 22, WAIT_HALO_G_EPILOGUE = 23,                                    // conv_halo.cuh
  WAIT_PAIR_FD_PRODUCER = 24, WAIT_PAIR_FD_MMA = 25, WAIT_PAIR_FD_EPILOGUE = 26,                                 // gemm2q.cuh
  WAIT_WIDE_PRODUCER = 31, WAIT_WIDE_MMA = 32, WAIT_WIDE_EPILOGUE = 33,                                          // conv_wide.cuh
  WAIT_CODE_MAX = 33
};

// Words of a status block: the code, then where that role stood.
enum { STATUS_CODE = 0, STATUS_CTA = 1, STATUS_TILE = 2, STATUS_STEP = 3, STATUS_WORDS = 4 };

constexpr const char* wait_code_name(int code) {
  return code <= 0                     ? "none"
         : code <= WAIT_GEMM_CHUNK     ? "single-CTA contraction"
         : code <= WAIT_CLUSTER_EPILOGUE ? "contraction divided over a cluster"
         : code <= WAIT_HALO_EPILOGUE  ? "halo-tile convolution"
         : code <= WAIT_PAIR_CHUNK     ? "SM-pair contraction"
         : code <= WAIT_PAIR_G_CHUNK   ? "persistent SM-pair G"
         : code <= WAIT_HALO_G_EPILOGUE ? "halo-tile G"
         : code <= WAIT_PAIR_FD_EPILOGUE ? "persistent SM-pair contraction"
         : code <= WAIT_CODE_MAX       ? "wide halo-tile convolution"
                                       : "unknown";
}
constexpr const char* wait_code_role(int code) {
  switch (code) {
    case WAIT_GEMM_PRODUCER: case WAIT_CLUSTER_PRODUCER: case WAIT_HALO_PRODUCER: case WAIT_PAIR_PRODUCER:
    case WAIT_PAIR_G_PRODUCER: case WAIT_HALO_G_PRODUCER: case WAIT_PAIR_FD_PRODUCER: case WAIT_WIDE_PRODUCER: return "producer";
    case WAIT_GEMM_MMA: case WAIT_CLUSTER_MMA: case WAIT_HALO_MMA: case WAIT_PAIR_MMA: case WAIT_PAIR_G_MMA:
    case WAIT_HALO_G_MMA: case WAIT_PAIR_FD_MMA: case WAIT_WIDE_MMA: return "MMA issuer";
    case WAIT_PAIR_G_UPDATE_PRODUCER: return "update-tile producer";
    case WAIT_GEMM_CHUNK: case WAIT_PAIR_CHUNK: case WAIT_PAIR_G_CHUNK: return "epilogue (update chunk)";
    default: return "epilogue";
  }
}

#ifdef __CUDACC__
// The first role that gives up writes the word and where it stood: the CTA, its tile, and the k-block (or update chunk).
__device__ __forceinline__ void report_expired(int* status, int code, int tile, int step) {
  if (atomicCAS(status + STATUS_CODE, 0, code) != 0) return;
  status[STATUS_CTA] = int(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z));
  status[STATUS_TILE] = tile;
  status[STATUS_STEP] = step;
}
#endif

}  // namespace lp
