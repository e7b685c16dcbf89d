// mpbp_alg1.cu -- beside Alg. 1's iteration: the illumination map behind its
// final threshold, and the copies of the Adam moments for checkpoints.
#include "aux_launch.h"

namespace mpbp {

namespace {

// one thread per (frame, frame pixel): out(s_j + k) += |P_m(k)|^2
__global__ void illumination_kernel(IllumArgs a) {
  const long long mm = (long long)a.m * a.m;
  const long long n = (long long)a.nframes * mm;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long f = i / mm, k = i - f * mm;
    const int mk = (int)(f / a.J), j = (int)(f - (long long)mk * a.J);
    const int k0 = (int)(k / a.m), k1 = (int)(k - (long long)k0 * a.m);
    const int r0 = a.scan[j].x + k0, r1 = a.scan[j].y + k1;
    if (r0 < 0 || r0 >= a.n1 || r1 < 0 || r1 >= a.n2) continue;
    const long long pi = a.probe_stride >= 0 ? mk * a.probe_stride
                         : (a.probe_stride == kProbePerFrame ? f : j) * mm;
    const float2 P = reinterpret_cast<const float2*>(a.probe)[pi + k];
    atomicAdd(a.out + (long long)r0 * a.n2 + r1, P.x * P.x + P.y * P.y);
  }
}

// blockIdx.y: which of the six arrays (a minibatch loop that resumes and saves
// is bound by the host's launches: 12 copies of 2 us each became two launches)
__global__ void moment_copy_kernel(const __grid_constant__ MomentCopy a) {
  uint32_t* const d = a.dst[blockIdx.y];
  const uint32_t* const q = a.src[blockIdx.y];
  const long long n = a.words[blockIdx.y], stride = (long long)gridDim.x * blockDim.x;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (((reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(q)) & 15) == 0) {
    const long long n4 = n / 4;
    for (long long k = i; k < n4; k += stride)
      reinterpret_cast<uint4*>(d)[k] = reinterpret_cast<const uint4*>(q)[k];
    i += 4 * n4;   // what is left
  }
  for (; i < n; i += stride) d[i] = q[i];
}

}  // namespace

cudaError_t launch_moment_copy(const MomentCopy& a, int num_sms, cudaStream_t s) {
  long long most = 1;
  for (long long w : a.words) most = w > most ? w : most;
  const long long b = (most + 1023) / 1024;
  moment_copy_kernel<<<dim3((unsigned)(b < num_sms * 2 ? b : num_sms * 2), 6), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_illumination(const IllumArgs& a, int num_sms, cudaStream_t s) {
  const long long n = (long long)a.nframes * a.m * a.m;
  const long long b = (n + 255) / 256;
  illumination_kernel<<<(int)(b < num_sms * 16 ? b : num_sms * 16), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace mpbp
