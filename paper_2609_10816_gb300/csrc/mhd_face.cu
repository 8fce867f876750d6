// mhd_face.cu -- face-sweep kernels of the single-box step (body in mhd_face.cuh).
#include <algorithm>

#include "mhd_face.cuh"

namespace mhd {

// one direction, one thread per segment (the form without work cursors: mhd_step_noalloc)
template <int RC, int RS>
__global__ void __launch_bounds__(kFaceThreads, kFaceMinBlocks) k_face(Dev D, int dir, int seg) {
  Line ln;
  int m0, m1;
  if (!sweep_line(D, dir, seg, ln, m0, m1)) return;
  face_piece<RC, RS>(D, dir, false, ln, m0, m1, LaneWalk{0, 0, 0}, true);
}

// The three face sweeps of a stage as one persistent launch: the segments of the x, y and z
// sweeps form one work list behind one cursor, so that the grid drains one tail per stage instead
// of one per direction (a warp takes 32 segments of up to 64 faces at a time, and the last ones
// run while the other SMs idle). A warp's 32 segments lie on an 8 x 4 patch of lines where the box
// allows (sweep_line_at), so that its lanes take the same Riemann-fan branch more often. Each
// direction's part of the list starts at a multiple of 32, so that an item of a lane sweep is one
// warp's.
__device__ __forceinline__ long long round32(long long t) { return (t + 31) / 32 * 32; }
template <int RC, int RS>
__global__ void __launch_bounds__(kFaceThreads, kFaceMinBlocks) k_faces(Dev D, int s0, int s1, int s2, int x_lanes) {
  const long long t0 = x_lanes ? lane_threads(D, 0, s0) : round32(sweep_threads(D, 0, s0));
  const long long t1 = round32(sweep_threads(D, 1, s1)), t2 = round32(sweep_threads(D, 2, s2));
  for_each_segment(work_cursor(D, CUR_FACE), t0 + t1 + t2, [&](long long t) {
    int dir = 0, seg = s0;
    if (t >= t0) {
      t -= t0;
      dir = 1;
      seg = s1;
      if (t >= t1) {
        t -= t1;
        dir = 2;
        seg = s2;
      }
    }
    face_thread<RC, RS>(D, dir, x_lanes && dir == 0, seg, t);
  });
}

// Boxes below this many cells walk the x sweep too: they have too few segments to pay for the pass
// that fills a lane sweep's windows (32^3, PLM + HLL: face sweeps of a step 114 us walked, 151 by
// lanes; 64^3, PPM + HLLD, one stage with stored states: 388 against 384).
constexpr long long kLaneCells = 1LL << 17;
// Points per segment of a walked face sweep: fill_seg's, and less for boxes that leave the GPU idle,
// though each segment starts its windows anew: a face in a walk waits for the one before it (about 7 us
// each on an idle GPU; face sweeps of a PPM + HLLD step with 4, 2 and 1: 8^3 104, 67, 48 us; 24^3 108,
// 88, 74; 32^3 144, 112, 128; 48^3 324, 292, 332).
static int walk_seg(const Dev& d, int dir, int seg, long long resident_threads) {
  int s = fill_seg(d, dir, seg, resident_threads);
  if (s <= 4 && sweep_threads(d, dir, 2) <= resident_threads) s = 2;
  if (s <= 2 && 3 * sweep_threads(d, dir, 1) <= resident_threads) s = 1;
  return s;
}
template <int RC, int RS>
static void launch_faces_t(const Dev& d, int seg, cudaStream_t st) {
  const int bs = kFaceThreads, smem = face_smem_bytes<RC>();
  const long long res = resident_blocks((const void*)k_faces<RC, RS>, bs, smem);
  int sg[3];
  long long tot = 0;
  const bool x_lanes = face_by_lanes(d, 0) && d.N >= kLaneCells;
  for (int dir = 0; dir < 3; ++dir) {
    if (dir == 0 && x_lanes) {
      // whole passes of 8; two items per resident warp, as fill_seg does for the others
      sg[dir] = lane_seg(2 * seg);
      while (sg[dir] > 8 && lane_threads(d, dir, sg[dir]) < 2 * res * bs) sg[dir] = lane_seg(sg[dir] / 2);
      tot += lane_threads(d, dir, sg[dir]);
    } else {
      sg[dir] = walk_seg(d, dir, seg, res * bs);
      tot += sweep_threads(d, dir, sg[dir]) + 31;
    }
  }
  const long long blocks = std::min((tot + bs - 1) / bs, res);
  k_faces<RC, RS><<<(unsigned)blocks, bs, smem, st>>>(d, sg[0], sg[1], sg[2], x_lanes ? 1 : 0);
}

template <int RC, int RS>
static void launch_face_t(const Dev& d, int dir, int seg, cudaStream_t st) {
  const int bs = kFaceThreads, smem = face_smem_bytes<RC>();
  // (the call also allows the kernel its shared memory. Segments of 64 faces whatever the box left its
  // chains of steps too long: mhd_step_noalloc at 32^3, PC + LLF 1.59 ms, so 0.47; PPM + HLLD 0.78, 4.03
  // with the windows in registers)
  const long long res = resident_blocks((const void*)k_face<RC, RS>, bs, smem);
  const int sg = walk_seg(d, dir, seg, res * bs);
  const long long threads = sweep_threads(d, dir, sg);
  k_face<RC, RS><<<(unsigned)((threads + bs - 1) / bs), bs, smem, st>>>(d, dir, sg);
}

template <int RC>
static void launch_face_r(const Dev& d, int dir, int rs, int seg, cudaStream_t st) {
  if (dir < 0) {  // all three directions in one launch
    switch (rs) {
      case RS_HLL: launch_faces_t<RC, RS_HLL>(d, seg, st); break;
      case RS_HLLD: launch_faces_t<RC, RS_HLLD>(d, seg, st); break;
      default: launch_faces_t<RC, RS_LLF>(d, seg, st); break;
    }
    return;
  }
  switch (rs) {
    case RS_HLL: launch_face_t<RC, RS_HLL>(d, dir, seg, st); break;
    case RS_HLLD: launch_face_t<RC, RS_HLLD>(d, dir, seg, st); break;
    default: launch_face_t<RC, RS_LLF>(d, dir, seg, st); break;
  }
}

void launch_face(const Dev& d, int dir, int recon, int rs, int seg, cudaStream_t st) {
  switch (recon) {
    case REC_PC: launch_face_r<REC_PC>(d, dir, rs, seg, st); break;
    case REC_PLM_MC: launch_face_r<REC_PLM_MC>(d, dir, rs, seg, st); break;
    case REC_PLM_MINMOD: launch_face_r<REC_PLM_MINMOD>(d, dir, rs, seg, st); break;
    case REC_PPM: launch_face_r<REC_PPM>(d, dir, rs, seg, st); break;
    default: launch_face_r<REC_PPM_EP>(d, dir, rs, seg, st); break;
  }
}

int launch_faces(const Dev& d, int recon, int rs, int seg, cudaStream_t st) {
  if (!d.work) {  // no work cursors: one launch per direction, one thread per segment
    for (int dir = 0; dir < 3; ++dir) launch_face(d, dir, recon, rs, seg, st);
    return 3;
  }
  launch_face(d, -1, recon, rs, seg, st);
  return 1;
}

}  // namespace mhd
