// mhd_face.cuh -- face sweep (Sec. 2.2): reconstruction along d + Riemann solve on every d-face,
// the Eq. (alpha-pm) speeds, the Q26 face velocity (Eq. q26-facevel), and the Joule energy flux of
// the Ohmic EMF (Sec. 2.4). One thread walks a segment of a periodic line along d; the
// reconstruction's sliding windows (Rec<> in mhd_device.cuh) move along with it, so each
// cell's slope, interface value and limiter are evaluated once per direction and each face's
// Riemann problem once, with no halo recomputation.
//
// What bounds it: the FP64 pipe (a warp instruction takes 64 cycles of it), then the latency of the
// integer instructions, loads and FP64 results between its instructions. The seven windows (49
// doubles of PPM) therefore sit in shared memory, not in registers, which lets 12 warps share an SM
// instead of the 8 that 255 registers allow; the loop over the seven variables is not unrolled (one
// copy of the reconstruction's code, no spills), and their states reach the solve through two more
// slots. An x sweep's lanes, each walking a line of its own, use 8 bytes of a 32-byte sector per
// step, and the sectors leave the caches before their next use: with 16 warps a 160^3 launch read
// 7.2 GB where 1.3 would do. Larger boxes therefore take the x sweep as a lane sweep, whose loads
// and stores cover whole sectors.
// Measured (face sweeps of a step; before / windows in registers, all unrolled; then as here with
// the x sweep walked; by lanes): 256^3 turbulence PPM + HLLD 30.6, 22.8, 21.0 ms; 128^3 with the
// FS18 EMF's extra stores 4.7, 3.9, 2.9 ms. With the two-instruction reciprocals 19.5 and 2.6: 98 to
// 107 FP64 warp instructions per 32 faces in 9.9 ms a launch at 256^3, about 77 cycles of their pipe
// each, where a fused multiply-add alone takes 64, an add or a product 76, and this mix (a third fused)
// 72.
#pragma once
#include "mhd_device.cuh"
#include "mhd_index.cuh"
#include "mhd_internal.cuh"

namespace mhd {

// Joule flux eta (j x b)_d on the d-face of cell X (reading: eta j from the mean of the face's
// two bounding edges per tangential direction, tangential b from the four nearest faces, which is
// the mean of the two cells' b). The edges' eta j / 2 were left with the primitives (store_current).
__device__ __forceinline__ double joule_flux(const Dev& D, int d, long long X) {
  const int a = (d + 1) % 3, c = (d + 2) % 3;
  const double* Ja = D.Epart + a * D.N;
  const double* Jc = D.Epart + c * D.N;
  const double* ba = D.P + (5 + a) * D.N;
  const double* bc = D.P + (5 + c) * D.N;
  const long long Xc = shift(D, X, c, 1), Xa = shift(D, X, a, 1), Xmd = shift(D, X, d, -1);
  const double ea = Ja[X] + Ja[Xc], ec = Jc[X] + Jc[Xa];
  const double bcbar = halve(bc[Xmd] + bc[X]), babar = halve(ba[Xmd] + ba[X]);
  return fma(ea, bcbar, -(ec * babar));
}

// The reconstruction windows of a block's threads in shared memory: slot k of variable v of a
// thread at (7 k + v) kFaceThreads + its number; the last two slots hand the face's left and right
// values to the solve.
constexpr int kFaceThreads = 128;
constexpr int kFaceMinBlocks = 3;  // blocks per SM (see above)
template <int RC>
constexpr int face_smem_bytes() {
  return (Rec<RC>::NS + 2) * 7 * kFaceThreads * (int)sizeof(double);
}

// The face at X with left and right states Lv, Rv in the face frame (n, t1, t2): rho, u_n, u_t1,
// u_t2, p, b_t1, b_t2. Solves it and stores fluxes, speeds and face velocity.
template <int RS>
__device__ __forceinline__ void face_solve(const Dev& D, int dir, long long X, const double* Lv, const double* Rv) {
  const int a = (dir + 1) % 3, c = (dir + 2) % 3;
  const long long N = D.N;
  // flux slots in the face frame: mass, the three momenta, energy
  double* F = D.F + 5LL * dir * N + X;
  double* const Fs[5] = {F, F + (1 + dir) * N, F + (1 + a) * N, F + (1 + c) * N, F + 4 * N};
  double Fold[5];  // stage 2: the stage-1 flux, on its way during the solve
  if (D.combine) {
#pragma unroll
    for (int v = 0; v < 5; ++v) Fold[v] = *Fs[v];
  }
  if (D.LR) {
    double* lr = D.LR + 14LL * dir * N;
#pragma unroll
    for (int v = 0; v < 7; ++v) {
      lr[v * N + X] = Lv[v];
      lr[(7 + v) * N + X] = Rv[v];
    }
  }
  if (D.emf == EMF_FS18) {
    double* VL = D.VL + 3LL * dir * N;
    double* VR = D.VR + 3LL * dir * N;
    VL[dir * N + X] = Lv[1]; VR[dir * N + X] = Rv[1];
    VL[a * N + X] = Lv[2];   VR[a * N + X] = Rv[2];
    VL[c * N + X] = Lv[3];   VR[c * N + X] = Rv[3];
  }
  const FaceState sl = {Lv[0], Lv[1], Lv[2], Lv[3], Lv[4], Lv[5], Lv[6]};
  const FaceState sr = {Rv[0], Rv[1], Rv[2], Rv[3], Rv[4], Rv[5], Rv[6]};
  double f[5], ap, am, us = 0.0;
  riemann<RS>(sl, sr, D.Bin[dir][X], D.gam, D.gm1inv, f, ap, am, us, D.emf == EMF_Q26);
  D.Ap[dir * N + X] = ap;
  D.Am[dir * N + X] = am;
  if (D.emf == EMF_Q26) D.Us[dir * N + X] = us;
  if (D.resistive) f[4] += joule_flux(D, dir, X);
  if (D.combine) {
#pragma unroll
    for (int v = 0; v < 5; ++v) *Fs[v] = halve(Fold[v] + f[v]);
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) *Fs[v] = f[v];
  }
}
// the rows of D.P in the face frame, four bits each
__device__ __forceinline__ unsigned face_rows(int dir) {
  const int a = (dir + 1) % 3, c = (dir + 2) % 3;
  return (unsigned)((1 + dir) << 4 | (1 + a) << 8 | (1 + c) << 12 | 4 << 16 | (5 + a) << 20 | (5 + c) << 24);
}

// One piece of a face sweep, in one of two forms that share the code of the solve (one copy of it in
// the kernel: a launch on a small box spends much of its time fetching instructions).
// A walk: the thread takes the faces m0 .. m1 - 1 of its line one after the other.
// A lane sweep (by_lanes; the warp's 32 threads call it together): 8 consecutive faces of 4 lines per
// pass, the thread's line being one of them (`active`: it exists), from a pass before m0, which only
// fills the windows. Along x a warp's lanes lie in rows of 8 on 4 lines (64 contiguous bytes of each).
template <int RC, int RS>
__device__ __forceinline__ void face_piece(const Dev& D, int dir, bool by_lanes, const Line& ln, int m0, int m1,
                                           const LaneWalk& w, bool active) {
  extern __shared__ double face_smem[];
  using LR = LaneRec<RC>;
  constexpr int LB = Rec<RC>::LB, LA = Rec<RC>::LA, NS = Rec<RC>::NS, NB = Rec<RC>::NB;
  constexpr int ST = 7 * kFaceThreads;  // stride of a variable's slots
  double* const win = face_smem + threadIdx.x;
  const long long N = D.N;
  const unsigned rows = face_rows(dir);
  unsigned codes = 0;
  if (!by_lanes) {
#pragma unroll 1
    for (int v = 0; v < 7; ++v) {
      const double* q = D.P + ((rows >> (4 * v)) & 7) * N;
      double p[LB + LA];
#pragma unroll
      for (int t = 0; t < LB + LA; ++t) p[t] = q[ln.at(m0 - LB + t)];
      Rec<RC> r;
      r.code = 0;
      r.template init<true>(p);
      r.each([&](int k, double& x) { win[k * ST + v * kFaceThreads] = x; });
      if (NB > 0) codes |= (unsigned)r.code << (NB * v);
    }
  } else {
#pragma unroll 1
    for (int k = 0; k < 7 * LR::NP; ++k) win[k * kFaceThreads] = 0.0;
  }
  int posN = by_lanes ? 0 : (m0 + LA) % ln.n;  // the point that enters a walk's windows
  const int inc = by_lanes ? 8 : 1;
  for (int mc = by_lanes ? m0 - 8 : m0; mc < m1; mc += inc) {
    const int m = by_lanes ? mc + w.k : mc;
    unsigned ncodes = 0;
    if (by_lanes) {
      // (m - 1 .. m + 2 lie within a line's length of [0, n): n >= 16)
      long long off[LR::NQ];
#pragma unroll
      for (int t = 0; t < LR::NQ; ++t) {
        int p = m + LR::FIRST + t;
        p += p < 0 ? ln.n : (p >= ln.n ? -ln.n : 0);
        off[t] = ln.base + (long long)p * ln.stride;
      }
      double qn[LR::NQ];
#pragma unroll
      for (int t = 0; t < LR::NQ; ++t) qn[t] = D.P[off[t]];  // (rows starts with rho's)
#pragma unroll 1
      for (int v = 0; v < 7; ++v) {
        double* const slot = win + v * kFaceThreads;
        double q[LR::NQ], prev[LR::NP > 0 ? LR::NP : 1], lv, rv;
#pragma unroll
        for (int t = 0; t < LR::NQ; ++t) q[t] = qn[t];
        if (v < 6) {  // on their way during this variable's step
          const double* const P = D.P + ((rows >> (4 * v + 4)) & 7) * N;
#pragma unroll
          for (int t = 0; t < LR::NQ; ++t) qn[t] = P[off[t]];
        }
#pragma unroll
        for (int k = 0; k < LR::NP; ++k) prev[k] = slot[k * ST];
        int code = NB > 0 ? (int)(codes >> (NB * v)) & ((1 << NB) - 1) : 0;
        LR::step(w, q, prev, code, lv, rv);
#pragma unroll
        for (int k = 0; k < LR::NP; ++k) slot[k * ST] = prev[k];
        slot[NS * ST] = lv;
        slot[(NS + 1) * ST] = rv;
        if (NB > 0) ncodes |= (unsigned)code << (NB * v);
      }
    } else {
      const double* const P = D.P + ln.base + (long long)posN * ln.stride;
      if (++posN == ln.n) posN = 0;
      double qn = P[0];
#pragma unroll 1
      for (int v = 0; v < 7; ++v) {
        double* const slot = win + v * kFaceThreads;
        Rec<RC> r;
        r.code = NB > 0 ? (int)(codes >> (NB * v)) & ((1 << NB) - 1) : 0;
        r.each([&](int k, double& x) { x = slot[k * ST]; });
        const double q = qn;
        if (v < 6) qn = P[((rows >> (4 * v + 4)) & 7) * N];
        double lv, rv;
        r.template step<true>(q, lv, rv);
        r.each([&](int k, double& x) { slot[k * ST] = x; });
        slot[NS * ST] = lv;
        slot[(NS + 1) * ST] = rv;
        if (NB > 0) ncodes |= (unsigned)r.code << (NB * v);
      }
    }
    codes = ncodes;
    if (m >= m0 && m < m1 && active) {
      double Lv[7], Rv[7];
#pragma unroll
      for (int v = 0; v < 7; ++v) {
        Lv[v] = win[NS * ST + v * kFaceThreads];
        Rv[v] = win[(NS + 1) * ST + v * kFaceThreads];
      }
      face_solve<RS>(D, dir, ln.base + (long long)m * ln.stride, Lv, Rv);
    }
    if (by_lanes) __syncwarp();
  }
}

// The line and place of this thread in item `item` of the lane sweep along dir (lane_threads).
__device__ __forceinline__ bool lane_line(const Dev& D, int dir, int seg, long long item, Line& ln, int& m0, int& m1,
                                          LaneWalk& w) {
  const int lane = threadIdx.x & 31;
  const bool x = dir == 0;
  w.k = x ? lane & 7 : lane >> 2;
  const int sub = x ? lane >> 3 : lane & 3;
  const int k1 = (w.k + 7) & 7, k2 = (w.k + 6) & 7;
  w.src1 = x ? (sub << 3) + k1 : (k1 << 2) + sub;
  w.src2 = x ? (sub << 3) + k2 : (k2 << 2) + sub;
  int t1, t2;
  sweep_axes(dir, t1, t2);
  const int groups = (int)lane_groups(D, dir), sidx = (int)(item / groups);
  const int nlines = D.n[t1] * D.n[t2];
  const int line = (int)(item - (long long)sidx * groups) * 4 + sub, l = min(line, nlines - 1);
  ln.base = (long long)(l % D.n[t1]) * D.stride[t1] + (long long)(l / D.n[t1]) * D.stride[t2];
  ln.stride = D.stride[dir];
  ln.n = D.n[dir];
  m0 = sidx * seg;
  m1 = min(ln.n, m0 + seg);
  return line < nlines;
}

// Thread t of the sweep along dir, cut into segments of seg faces.
template <int RC, int RS>
__device__ __forceinline__ void face_thread(const Dev& D, int dir, bool by_lanes, int seg, long long t) {
  Line ln;
  LaneWalk w = {0, 0, 0};
  int m0, m1;
  bool active;
  if (by_lanes) {
    active = lane_line(D, dir, seg, t >> 5, ln, m0, m1, w);
  } else {
    active = sweep_line_at(D, dir, seg, t, ln, m0, m1, false, true);
    if (!active) return;
  }
  face_piece<RC, RS>(D, dir, by_lanes, ln, m0, m1, w, active);
}

// Whether the sweep along dir runs as a lane sweep: along x, on lines of at least 16 points with at
// most a sixteenth of the lanes idle in a line's last pass, and of those in the last group of 4 lines
// (2^22 cells, PPM + HLLD step, by lanes and walked: 1 line 20.2 and 13.2 ms, 2 lines 16.1 and 13.7, 5
// lines 14.1 and 12.8, 13 lines 13.2 and 13.1, 26 lines 13.7 and 14.0, 64 x 64 lines 11.9 and 12.4).
__host__ __device__ __forceinline__ bool face_by_lanes(const Dev& D, int dir) {
  const int n = D.n[dir];
  const long long lines = (long long)D.n[1] * D.n[2];
  return dir == 0 && n >= 16 && (n + 7) / 8 * 120LL <= 16LL * n && (lines + 3) / 4 * 60 <= 16 * lines;
}

}  // namespace mhd
