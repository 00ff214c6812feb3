// rm_mesh.cu -- rm_meshify: the labelled interface mesh of one range image (Sec. IV.A, Fig. 5).
//
// Two kernels (three for large images), in a fixed order so that the output is the same run to run
// (row-major block order, no atomics):
//   k_mesh_blocks  per grid pixel: the world vertex through the pose in FP64 (rounded once to
//                  FP32); per 2x2 block of grid pixels: dropped when a pixel is dead, else FU when
//                  a pixel is a no-return or a side or the diagonal is longer than the limit
//                  (squared lengths in FP32), else FO; plus the kept count of each CTA. The
//                  camera-frame points of a block's corners are computed again for each block
//                  rather than kept: their inputs are in L1.
//   k_mesh_scan    large images only (more than kScanCtas CTAs): exclusive scan of the counts
//   k_mesh_emit    per block: two triangles (v00, v10, v11), (v00, v11, v01) at the block's
//                  rank among the kept blocks; each CTA adds up the counts before its own
// The arithmetic that decides a label uses explicitly rounded operations (no contraction), so
// the decision is the same as any IEEE FP32 evaluation in the same order. One 640x480 image is
// launches and latency: 352 -> 130 us a call, most of it the scratch that used to be allocated
// and, at the call's synchronisation, given back to the system each time.
#include <cfloat>
#include <cmath>
#include <string>

#include "rendermap.h"
#include "rm_kernels.cuh"

namespace {

constexpr int kQuadThreads = 256;

struct MeshArgs {
  int model, W, H, step, Ws, Hs;
  float fx, fy, cx, cy;
  const float *rays;
  const float *depth;
  const uint8_t *cls;
  double T[12];         // camera-to-world rows (R | t) of a host pose
  const double *Tdev;   // or the pose in device memory (16 doubles)
  float max_range, lim;  // lim = max_edge^2 (FP32)
  float *vertices;
  uint8_t *qcode;       // per block: 0 dropped, 1 FO, 2 FU
  int *cta_count;
  long long *cta_off;   // exclusive offsets (in blocks), or null: k_mesh_emit adds up cta_count
  int n_cta;            // CTAs that hold blocks
  int32_t *faces;
  uint8_t *labels;
  long long *n_faces;
};

// Up to here every CTA of k_mesh_emit adds up the counts before its own: half of n^2 integers in
// all, 8 MB from L2 at this line, less than the scan's launch (3.8 us) costs at 1200 CTAs; the sums
// grow with the square from there.
constexpr int kScanCtas = 2048;

// Kind (0 return, 1 no-return, 2 dead) and camera-frame point of grid pixel (i, j).
__device__ __forceinline__ int mesh_point(const MeshArgs &a, int i, int j, float3 &pc) {
  const int x = i * a.step, y = j * a.step;
  const long long p = (long long)y * a.W + x;
  const float d = __ldg(a.depth + p);
  const int c = __ldg(a.cls + p);
  const int k = (c > 1 || !(fabsf(d) <= FLT_MAX)) ? 2 : c;
  const float r = k == 0 ? d : (k == 1 ? a.max_range : 0.0f);
  float rx, ry, rz;
  if (a.model == RM_PINHOLE) {
    rx = __fdiv_rn(__fsub_rn(__fadd_rn((float)x, 0.5f), a.cx), a.fx);
    ry = __fdiv_rn(__fsub_rn(__fadd_rn((float)y, 0.5f), a.cy), a.fy);
    rz = 1.0f;
  } else {
    const float *q = a.rays + 3 * p;
    rx = q[0];
    ry = q[1];
    rz = q[2];
  }
  pc = make_float3(__fmul_rn(r, rx), __fmul_rn(r, ry), __fmul_rn(r, rz));
  return k;
}

__device__ __forceinline__ float edge2(const float3 &a, const float3 &b) {
  const float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y), dz = __fsub_rn(a.z, b.z);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// Thread v: grid pixel v, which is the first corner of a block unless it ends its row or column.
__global__ void __launch_bounds__(kQuadThreads) k_mesh_blocks(MeshArgs a) {
  const long long v = (long long)blockIdx.x * kQuadThreads + threadIdx.x;
  const bool on = v < (long long)a.Ws * a.Hs;
  const int i = on ? (int)(v % a.Ws) : 0, j = on ? (int)(v / a.Ws) : 0;
  int code = 0;
  if (on) {
    float3 A;
    const int k00 = mesh_point(a, i, j, A);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double *m = (a.Tdev ? a.Tdev : a.T) + 4 * q;
      double w = m[3];  // dead pixels stay at the sensor origin (unreferenced)
      if (k00 != 2)
        w = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(m[0], (double)A.x), __dmul_rn(m[1], (double)A.y)),
                                __dmul_rn(m[2], (double)A.z)),
                      m[3]);
      a.vertices[3 * v + q] = (float)w;
    }
    if (i + 1 < a.Ws && j + 1 < a.Hs) {
      float3 B, C, D;
      const int k10 = mesh_point(a, i + 1, j, B), k11 = mesh_point(a, i + 1, j + 1, C), k01 = mesh_point(a, i, j + 1, D);
      if (k00 != 2 && k10 != 2 && k01 != 2 && k11 != 2) {
        const bool fu = k00 == 1 || k10 == 1 || k01 == 1 || k11 == 1 || edge2(A, B) > a.lim || edge2(B, C) > a.lim ||
                        edge2(C, D) > a.lim || edge2(D, A) > a.lim || edge2(A, C) > a.lim;
        code = fu ? 2 : 1;
      }
    }
    a.qcode[v] = (uint8_t)code;
  }
  const int kept = __syncthreads_count(code != 0);
  if (threadIdx.x == 0) a.cta_count[blockIdx.x] = kept;
}

__global__ void __launch_bounds__(1024) k_mesh_scan(MeshArgs a) {
  __shared__ long long carry;
  __shared__ long long wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < a.n_cta; base += 1024) {
    const int idx = base + threadIdx.x;
    const long long c = idx < a.n_cta ? a.cta_count[idx] : 0;
    long long s = c;  // inclusive scan within the warp
    for (int off = 1; off < 32; off <<= 1) {
      const long long t = __shfl_up_sync(0xffffffffu, s, off);
      if (lane >= off) s += t;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
      long long w = wsum[lane];
      for (int off = 1; off < 32; off <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += t;
      }
      wsum[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    const long long before = carry + (warp > 0 ? wsum[warp - 1] : 0) + s - c;
    if (idx < a.n_cta) a.cta_off[idx] = before;
    __syncthreads();
    if (threadIdx.x == 1023) carry = before + c;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kQuadThreads) k_mesh_emit(MeshArgs a) {
  __shared__ int wcount[kQuadThreads / 32];
  __shared__ long long wbefore[kQuadThreads / 32];
  const long long v = (long long)blockIdx.x * kQuadThreads + threadIdx.x;
  const bool on = v < (long long)a.Ws * a.Hs;
  const int code = on ? a.qcode[v] : 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(0xffffffffu, code != 0);
  long long before = 0;  // kept blocks of the CTAs before this one
  if (!a.cta_off) {
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kQuadThreads) before += a.cta_count[k];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
  }
  if (lane == 0) {
    wcount[warp] = __popc(m);
    wbefore[warp] = before;
  }
  __syncthreads();
  int rank = __popc(m & ((1u << lane) - 1));
  for (int w = 0; w < warp; ++w) rank += wcount[w];
  if (a.cta_off) {
    before = a.cta_off[blockIdx.x];
  } else {
    before = 0;
    for (int w = 0; w < kQuadThreads / 32; ++w) before += wbefore[w];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kQuadThreads - 1) *a.n_faces = 2 * (before + rank + (code != 0));
  if (code == 0) return;
  const int v00 = (int)v, v10 = v00 + 1, v01 = v00 + a.Ws, v11 = v01 + 1;
  const long long f = 2 * (before + rank);
  int32_t *o = a.faces + 3 * f;
  o[0] = v00;
  o[1] = v10;
  o[2] = v11;
  o[3] = v00;
  o[4] = v11;
  o[5] = v01;
  const uint8_t lab = code == 2 ? 1 : 0;
  a.labels[f] = lab;
  a.labels[f + 1] = lab;
}

rm_status mf_fail(rm_status s, const std::string &m) {
  rmapi::set_error(m);
  return s;
}

}  // namespace

extern "C" rm_status rm_meshify(const rm_scan *scan, const double *pose,
                                const rm_meshify_params *prm, float *vertices, int32_t *faces,
                                uint8_t *labels, int64_t *n_faces, void *stream) {
  if (!scan || !pose || !prm || !n_faces) return mf_fail(RM_EINVAL, "NULL argument");
  if (!scan->depth || !scan->cls) return mf_fail(RM_EINVAL, "scan arrays are NULL");
  rm_status st = rmapi::check_intrinsics(&scan->intr);
  if (st != RM_OK) return st;
  if (prm->step < 1 || prm->step > 64) return mf_fail(RM_EINVAL, "step must be 1..64");
  if (!(prm->max_range > 0.0f) || !(prm->max_range <= FLT_MAX))
    return mf_fail(RM_EINVAL, "max_range must be finite and > 0");
  if (!(prm->max_edge >= 0.0f) || !(prm->max_edge <= FLT_MAX))
    return mf_fail(RM_EINVAL, "max_edge must be finite and >= 0");
  cudaStream_t s = (cudaStream_t)stream;
  // a host pose is checked here and passed by value; a device pose is read by the kernel in
  // place (no host round trip; a non-finite one gives non-finite vertices)
  const bool dev_pose = rmapi::is_device_pointer(pose);
  if (!dev_pose)
    for (int k = 0; k < 12; ++k)
      if (!std::isfinite(pose[k])) return mf_fail(RM_EINVAL, "pose must be finite");
  const rm_intrinsics &in = scan->intr;
  const int Ws = (in.width - 1) / prm->step + 1, Hs = (in.height - 1) / prm->step + 1;
  const long long NV = (long long)Ws * Hs, NQ = (long long)(Ws - 1) * (Hs - 1);
  if (!vertices || (NQ > 0 && (!faces || !labels))) return mf_fail(RM_EINVAL, "NULL output array");
  const long long P = (long long)in.width * in.height;
  const bool host_d = !rmapi::is_device_pointer(scan->depth), host_c = !rmapi::is_device_pointer(scan->cls);
  const bool host_r = in.model == RM_RAYTABLE && !rmapi::is_device_pointer(in.rays);
  const bool host_v = !rmapi::is_device_pointer(vertices);
  const bool host_f = NQ > 0 && !rmapi::is_device_pointer(faces);
  const bool host_l = NQ > 0 && !rmapi::is_device_pointer(labels);
  const bool host_n = !rmapi::is_device_pointer(n_faces);
  const int n_cta = (int)((NV + kQuadThreads - 1) / kQuadThreads);
  // one stream-ordered scratch block: staged inputs and outputs, then the work arrays
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t o_d = host_d ? take(sizeof(float) * P) : 0, o_c = host_c ? take(P) : 0;
  const size_t o_r = host_r ? take(sizeof(float) * 3 * P) : 0;
  const size_t o_v = host_v ? take(sizeof(float) * 3 * NV) : 0;
  const size_t o_f = host_f ? take(sizeof(int32_t) * 6 * NQ) : 0;
  const size_t o_l = host_l ? take(2 * NQ) : 0;
  const size_t o_q = take(NV), o_cc = take(sizeof(int) * n_cta);
  const size_t o_co = n_cta > kScanCtas ? take(sizeof(long long) * n_cta) : 0;
  const size_t o_n = take(sizeof(long long));
  unsigned char *buf = nullptr;
  cudaError_t e = rmapi::scratch_alloc((void **)&buf, off, s);
  if (e != cudaSuccess) return mf_fail(RM_ENOMEM, std::string("rm_meshify: ") + cudaGetErrorString(e));
  auto ck = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  MeshArgs a{};
  a.model = in.model;
  a.W = in.width;
  a.H = in.height;
  a.step = prm->step;
  a.Ws = Ws;
  a.Hs = Hs;
  a.fx = in.fx;
  a.fy = in.fy;
  a.cx = in.cx;
  a.cy = in.cy;
  a.depth = host_d ? reinterpret_cast<float *>(buf + o_d) : scan->depth;
  a.cls = host_c ? buf + o_c : scan->cls;
  a.rays = host_r ? reinterpret_cast<float *>(buf + o_r) : in.rays;
  for (int k = 0; k < 12; ++k) a.T[k] = dev_pose ? 0.0 : pose[k];
  a.Tdev = dev_pose ? pose : nullptr;
  a.max_range = prm->max_range;
  a.lim = prm->max_edge * prm->max_edge;
  a.vertices = host_v ? reinterpret_cast<float *>(buf + o_v) : vertices;
  a.qcode = buf + o_q;
  a.cta_count = reinterpret_cast<int *>(buf + o_cc);
  a.cta_off = n_cta > kScanCtas ? reinterpret_cast<long long *>(buf + o_co) : nullptr;
  a.n_cta = n_cta;
  a.faces = host_f ? reinterpret_cast<int32_t *>(buf + o_f) : faces;
  a.labels = host_l ? buf + o_l : labels;
  a.n_faces = host_n ? reinterpret_cast<long long *>(buf + o_n) : reinterpret_cast<long long *>(n_faces);
  if (host_d) ck(cudaMemcpyAsync((void *)a.depth, scan->depth, sizeof(float) * P, cudaMemcpyHostToDevice, s));
  if (host_c) ck(cudaMemcpyAsync((void *)a.cls, scan->cls, P, cudaMemcpyHostToDevice, s));
  if (host_r) ck(cudaMemcpyAsync((void *)a.rays, in.rays, sizeof(float) * 3 * P, cudaMemcpyHostToDevice, s));
  if (e == cudaSuccess) {
    k_mesh_blocks<<<n_cta, kQuadThreads, 0, s>>>(a);
    ck(cudaGetLastError());
  }
  if (e == cudaSuccess && a.cta_off) {
    k_mesh_scan<<<1, 1024, 0, s>>>(a);
    ck(cudaGetLastError());
  }
  if (e == cudaSuccess) {
    k_mesh_emit<<<n_cta, kQuadThreads, 0, s>>>(a);
    ck(cudaGetLastError());
  }
  long long nf = 0;
  if (e == cudaSuccess && (host_n || host_f || host_l)) {
    ck(cudaMemcpyAsync(&nf, a.n_faces, sizeof(long long), cudaMemcpyDeviceToHost, s));
    ck(cudaStreamSynchronize(s));
  }
  if (e == cudaSuccess && host_v) ck(cudaMemcpyAsync(vertices, a.vertices, sizeof(float) * 3 * NV, cudaMemcpyDeviceToHost, s));
  if (e == cudaSuccess && host_f && nf > 0)
    ck(cudaMemcpyAsync(faces, a.faces, sizeof(int32_t) * 3 * nf, cudaMemcpyDeviceToHost, s));
  if (e == cudaSuccess && host_l && nf > 0) ck(cudaMemcpyAsync(labels, a.labels, nf, cudaMemcpyDeviceToHost, s));
  cudaFreeAsync(buf, s);
  if (e == cudaSuccess && (host_v || host_f || host_l || host_n)) ck(cudaStreamSynchronize(s));
  if (e != cudaSuccess) return mf_fail(RM_ECUDA, std::string("rm_meshify: ") + cudaGetErrorString(e));
  if (host_n) *n_faces = nf;
  return RM_OK;
}
