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
// instead of the 8 that 255 registers allow: at 256^3 (turbulence, PPM + HLLD) the sweeps of a step
// take 23.2 ms with 3 blocks of 128 threads per SM and 23.5 with 2 (32.8 before). A fourth (128 registers, a few
// of them spilled) is slower, 29.9: an x sweep's lanes each walk a line of their own and use 8 bytes
// of a 32-byte sector per step, and with 16 warps the sectors leave the caches before their next
// use (7.2 GB read by a 160^3 launch that needs 1.3).
#pragma once
#include "mhd_device.cuh"
#include "mhd_index.cuh"
#include "mhd_internal.cuh"

namespace mhd {

// Joule flux eta (j x b)_d on the d-face of cell X (reading: eta j from the mean of the face's
// two bounding edges per tangential direction, tangential b from the four nearest faces).
__device__ __forceinline__ double joule_flux(const Dev& D, int d, long long X) {
  const int a = (d + 1) % 3, c = (d + 2) % 3;
  const double* Ba = D.Bin[a];
  const double* Bc = D.Bin[c];
  // j_e on the e-edge stored at Y: (B_{c_e}[Y] - B_{c_e}[Y - a_e]) / h_{a_e}
  //                               - (B_{a_e}[Y] - B_{a_e}[Y - c_e]) / h_{c_e}
  auto jedge = [&](int e, long long Y) {
    const int ae = (e + 1) % 3, ce = (e + 2) % 3;
    const double* Bce = D.Bin[ce];
    const double* Bae = D.Bin[ae];
    return (Bce[Y] - Bce[shift(D, Y, ae, -1)]) * D.hinv[ae] - (Bae[Y] - Bae[shift(D, Y, ce, -1)]) * D.hinv[ce];
  };
  const long long Xc = shift(D, X, c, 1), Xa = shift(D, X, a, 1), Xmd = shift(D, X, d, -1);
  const double ea = 0.5 * D.eta * (jedge(a, X) + jedge(a, Xc));
  const double ec = 0.5 * D.eta * (jedge(c, X) + jedge(c, Xa));
  const double bcbar = 0.25 * (Bc[Xmd] + Bc[X] + Bc[shift(D, Xmd, c, 1)] + Bc[Xc]);
  const double babar = 0.25 * (Ba[Xmd] + Ba[X] + Ba[shift(D, Xmd, a, 1)] + Ba[Xa]);
  return fma(ea, bcbar, -ec * babar);
}

// The reconstruction windows of a block's threads in shared memory: slot k of variable v of a
// thread at (7 k + v) kFaceThreads + its number.
constexpr int kFaceThreads = 128;
constexpr int kFaceMinBlocks = 3;  // blocks per SM (see above)
template <int RC>
constexpr int face_smem_bytes() {
  return Rec<RC>::NS * 7 * kFaceThreads * (int)sizeof(double);
}

template <int RC, int RS>
__device__ __forceinline__ void face_seg(const Dev& D, int dir, const Line& ln, int m0, int m1) {
  extern __shared__ double face_smem[];
  constexpr int LB = Rec<RC>::LB, LA = Rec<RC>::LA, NB = Rec<RC>::NB;
  constexpr int ST = 7 * kFaceThreads;  // stride of a variable's slots
  double* const win = face_smem + threadIdx.x;
  const int a = (dir + 1) % 3, c = (dir + 2) % 3;
  const long long N = D.N;
  // the primitives in the face frame (n, t1, t2): rho, u_n, u_t1, u_t2, p, b_t1, b_t2 (their rows of
  // D.P, four bits each)
  const unsigned rows = (unsigned)((1 + dir) << 4 | (1 + a) << 8 | (1 + c) << 12 | 4 << 16 | (5 + a) << 20 | (5 + c) << 24);
  unsigned codes = 0;
#pragma unroll 1
  for (int v = 0; v < 7; ++v) {
    const double* q = D.P + ((rows >> (4 * v)) & 7) * N;
    double w[LB + LA];
#pragma unroll
    for (int t = 0; t < LB + LA; ++t) w[t] = q[ln.at(m0 - LB + t)];
    Rec<RC> r;
    r.code = 0;
    r.init(w);
    r.each([&](int k, double& x) { win[k * ST + v * kFaceThreads] = x; });
    if (NB > 0) codes |= (unsigned)r.code << (NB * v);
  }
  // the point of the face, and the point that enters the windows with it
  long long Y = ln.at(m0);
  int posY = m0 % ln.n, posN = (m0 + LA) % ln.n;
  const bool fs18 = D.emf == EMF_FS18;
  for (int m = m0; m < m1; ++m) {
    const double* const P = D.P + ln.base + (long long)posN * ln.stride;
    double qn[7], Lv[7], Rv[7];
#pragma unroll
    for (int v = 0; v < 7; ++v) qn[v] = P[((rows >> (4 * v)) & 7) * N];
    unsigned ncodes = 0;
#pragma unroll
    for (int v = 0; v < 7; ++v) {
      double* const slot = win + v * kFaceThreads;
      Rec<RC> r;
      r.code = NB > 0 ? (int)(codes >> (NB * v)) & ((1 << NB) - 1) : 0;
      r.each([&](int k, double& x) { x = slot[k * ST]; });
      r.step(qn[v], Lv[v], Rv[v]);
      r.each([&](int k, double& x) { slot[k * ST] = x; });
      if (NB > 0) ncodes |= (unsigned)r.code << (NB * v);
    }
    codes = ncodes;
    // flux slots in the face frame (n, t1, t2): mass, the three momenta, energy
    double* F = D.F + 5LL * dir * N + Y;
    double Fold[5];  // stage 2: the stage-1 flux, on its way during the solve
    double* const Fs[5] = {F, F + (1 + dir) * N, F + (1 + a) * N, F + (1 + c) * N, F + 4 * N};
    if (D.combine) {
#pragma unroll
      for (int v = 0; v < 5; ++v) Fold[v] = *Fs[v];
    }
    if (D.LR) {
      double* lr = D.LR + 14LL * dir * N;
#pragma unroll
      for (int v = 0; v < 7; ++v) {
        lr[v * N + Y] = Lv[v];
        lr[(7 + v) * N + Y] = Rv[v];
      }
    }
    if (fs18) {
      double* VL = D.VL + 3LL * dir * N;
      double* VR = D.VR + 3LL * dir * N;
      VL[dir * N + Y] = Lv[1]; VR[dir * N + Y] = Rv[1];
      VL[a * N + Y] = Lv[2];   VR[a * N + Y] = Rv[2];
      VL[c * N + Y] = Lv[3];   VR[c * N + Y] = Rv[3];
    }
    const FaceState sl = {Lv[0], Lv[1], Lv[2], Lv[3], Lv[4], Lv[5], Lv[6]};
    const FaceState sr = {Rv[0], Rv[1], Rv[2], Rv[3], Rv[4], Rv[5], Rv[6]};
    double f[5], ap, am, us;
    riemann<RS>(sl, sr, D.Bin[dir][Y], D.gam, D.gm1inv, f, ap, am, us);
    D.Ap[dir * N + Y] = ap;
    D.Am[dir * N + Y] = am;
    D.Us[dir * N + Y] = us;
    if (D.resistive) f[4] += joule_flux(D, dir, Y);
    if (D.combine) {
#pragma unroll
      for (int v = 0; v < 5; ++v) *Fs[v] = halve(Fold[v] + f[v]);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) *Fs[v] = f[v];
    }
    if (++posY == ln.n) posY = 0;
    if (++posN == ln.n) posN = 0;
    Y = ln.base + (long long)posY * ln.stride;
  }
}

}  // namespace mhd
