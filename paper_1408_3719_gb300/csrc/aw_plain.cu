// The heavy sweep kernels in plain FP64, for differentiated runs (states loaded
// by aw_load_state_xy, and the sweeps of aw_adjoint_forward / aw_adjoint); all
// other runs take the faster kernels of aw_kernels.cu, which round differently.
//
// Why the gradients keep this rounding: the characteristic fields' direction is
// the density gradient over its length, also where a uniform flow's gradient is
// rounding noise, and its derivative divides by that noise.  The gradient of the
// whole mesh's kinetic energy on the isentropic vortex therefore moves by
// 2e-9..7e-7 of its norm (P1-P3, 1,800 to 49,928 triangles, 20 sweeps) when only
// the predictor's roundings change, while the run's own state moves by 1e-15;
// with these kernels it reproduces.
#include <algorithm>

#include "aw_internal.h"

namespace aw {

namespace {

// ---------------------------------------------------------------------------
// Cooperative predictor: one thread per (element, space-time node), G
// elements per 128-thread block, the element's nodal arrays in shared memory.
// ---------------------------------------------------------------------------
template <int M, int TH = 128>
struct PredShape {
  static constexpr int Mc = (M + 1) * (M + 2) / 2, Nt = M + 1, Nst = Mc * Nt;
  static constexpr int kThreads = TH;
  static constexpr int G = kThreads / Nst;
};

template <int M, int TH>
__global__ void __launch_bounds__(TH, TH >= 256 ? 2 : 3) k_predict_coop(Tab T, Dev d, int initial, int gts) {
  using S = PredShape<M, TH>;
  constexpr int Mc = S::Mc, Nt = S::Nt, Nst = S::Nst, G = S::G;
  __shared__ double sq[G][Nst][4], sf[G][Nst][4], sg[G][Nst][4], sP[G][Nst][4];
  __shared__ double sx[G][Nst][2], sV[G][Nst][2];
  // sTr: the 3 Nt rows of edge-trace weights (edge, Gauss point), then the
  // reference-average weights, so that traces and averages share one code path
  __shared__ double sDxi[Mc][Mc], sDeta[Mc][Mc], sB[Nt - 1][Nt], sDtau[Nt][Nt], sTr[3 * Nt + 1][Mc], sVt[Nt][Nt];
  __shared__ double sdts[G];
  __shared__ int sidx[G], sbad[G];
  for (int k = threadIdx.x; k < Mc * Mc; k += blockDim.x) {
    sDxi[k / Mc][k % Mc] = T.Dxi[k / Mc][k % Mc];
    sDeta[k / Mc][k % Mc] = T.Deta[k / Mc][k % Mc];
  }
  for (int k = threadIdx.x; k < (Nt - 1) * Nt; k += blockDim.x) sB[k / Nt][k % Nt] = T.B[k / Nt][k % Nt];
  for (int k = threadIdx.x; k < Nt * Nt; k += blockDim.x) {
    sDtau[k / Nt][k % Nt] = T.Dtau[k / Nt][k % Nt];
    sVt[k / Nt][k % Nt] = T.VtInv[k / Nt][k % Nt];
  }
  for (int k = threadIdx.x; k < 3 * Nt * Mc; k += blockDim.x) sTr[k / Mc][k % Mc] = T.Tr[k / (Nt * Mc)][(k / Mc) % Nt][k % Mc];
  for (int k = threadIdx.x; k < Mc; k += blockDim.x) sTr[3 * Nt][k] = T.wavg[k];
  const int n_ready = initial ? d.ne : d.cnt->n_ready;
  const long long gmin = d.cnt->gts_min;
  // thread -> (time slice t, element e, lattice node s).  A warp-wide FP64
  // instruction costs the FP64 pipe the same whatever number of its lanes is
  // active, so the tau = 0 nodes (full work in the first iteration only) and
  // the tau > 0 nodes (full work in the later ones) sit in separate warps:
  // the tau = 0 nodes of all G elements first, padded to a whole warp, when
  // that fits the block, otherwise after the tau > 0 nodes.
  constexpr int nBot = G * Mc, nTop = G * Mc * (Nt - 1), nBotPad = (nBot + 31) / 32 * 32;
  constexpr bool padBot = nBotPad + nTop <= TH;
  // When one element's tau > 0 nodes nearly fill a warp (30 of 32 lanes at
  // fourth order), each element gets a warp of its own: the warps of the
  // elements a round leaves empty (balanced rounds give a block fewer than G
  // elements) then issue no instruction at all.
  constexpr int nTopE = Mc * (Nt - 1);
  constexpr bool perWarp = nTopE > 16 && nTopE <= 32 && nBotPad + 32 * G <= TH;
  int t, rr;
  if (perWarp) {
    const int x = threadIdx.x;
    const int ew = (x - nBotPad) >> 5, k = (x - nBotPad) & 31;
    if (x < nBot) { t = 0; rr = x; }
    else if (x >= nBotPad && ew < G && k < nTopE) { t = 1 + k / Mc; rr = ew * Mc + k % Mc; }
    else { t = Nt; rr = 0; }
  } else if (padBot) {
    const int x = threadIdx.x;
    if (x < nBot) { t = 0; rr = x; }
    else if (x >= nBotPad && x < nBotPad + nTop) { t = 1 + (x - nBotPad) / nBot; rr = (x - nBotPad) % nBot; }
    else { t = Nt; rr = 0; }
  } else {
    const int x = threadIdx.x;
    if (x < nTop) { t = 1 + x / nBot; rr = x % nBot; }
    else if (x < nTop + nBot) { t = 0; rr = x - nTop; }
    else { t = Nt; rr = 0; }
  }
  const int e = t < Nt ? rr / Mc : G;
  const int s = rr % Mc, l = (t < Nt ? t : 0) * Mc + s;
  const double gm1 = T.gamma - 1.0;
  for (int consumed = 0; consumed < n_ready;) {
    // balanced rounds, as in the reconstruction
    const int per = min(G, (n_ready - consumed + (int)gridDim.x - 1) / (int)gridDim.x);
    const int base = consumed + (int)blockIdx.x * per;
    const int cnt = max(0, min(per, n_ready - base));
    consumed += per * (int)gridDim.x;
    if (cnt == 0) continue;  // block-uniform
    const int pos = base + e;
    const bool live = e < cnt;
    if (live && l == 0) {
      const int i = initial ? pos : d.ready_list[pos];
      long long dtk = d.dt[i];
      if ((gts || d.t[i] < T.Tsw) && dtk > 0) {
        dtk = gmin;
        d.dt[i] = dtk;
      }
      sidx[e] = i;
      sdts[e] = (double)dtk * d.etick[i];
      sbad[e] = 0;
    }
    __syncthreads();
    const int i = live ? sidx[e] : 0;
    const double dts = live ? sdts[e] : 0.0;
    const bool work = live && dts > 0.0;
    if (live) {
      const double* w0 = d.w0 + (size_t)pos * Mc * 4;
#pragma unroll
      for (int v = 0; v < 4; ++v) sq[e][l][v] = w0[s * 4 + v];
      const double* X = d.X + 6 * (size_t)i;
      sx[e][l][0] = X[0] + (X[2] - X[0]) * T.lat[s][0] + (X[4] - X[0]) * T.lat[s][1];
      sx[e][l][1] = X[1] + (X[3] - X[1]) * T.lat[s][0] + (X[5] - X[1]) * T.lat[s][1];
    }
    __syncthreads();
    const double idt = work ? 1.0 / dts : 0.0;
    // tau = 0 node: its data and spatial metric never change, so after the
    // first iteration only the xi_t, eta_t terms of P are recomputed there
    double c_fs[4] = {0, 0, 0, 0}, c_Qx[4] = {0, 0, 0, 0}, c_Qe[4] = {0, 0, 0, 0};
    double c_xix = 0, c_xiy = 0, c_etx = 0, c_ety = 0;
    for (int it = 0; it < T.nit; ++it) {
      // Iteration 0 starts from w_h at every slice and a static geometry, so P
      // is the same on every slice: it is computed on the tau = 0 slice only.
      const bool full = work && (it == 0 ? t == 0 : t > 0);
      if (full) {  // nodal fluxes and mesh velocity at the own node
        const double* q = sq[e][l];
        const double ir = 1.0 / q[0], u = q[1] * ir, v = q[2] * ir;
        const double p = gm1 * (q[3] - 0.5 * (q[1] * u + q[2] * v));
        sf[e][l][0] = q[1]; sf[e][l][1] = q[1] * u + p; sf[e][l][2] = q[1] * v; sf[e][l][3] = u * (q[3] + p);
        sg[e][l][0] = q[2]; sg[e][l][1] = q[2] * u; sg[e][l][2] = q[2] * v + p; sg[e][l][3] = v * (q[3] + p);
        sV[e][l][0] = T.eulerian ? 0.0 : u;
        sV[e][l][1] = T.eulerian ? 0.0 : v;
      }
      __syncthreads();
      if (full && t > 0) {
        // tau > 0 node (later iterations): P at the own node (eq. pdef) with
        // the isoparametric metric (eq. Jac) first, then one contraction with
        // the combined weights D_xi xi_x + D_eta eta_x (and the y, t ones)
        double xx = 0, xe = 0, yx = 0, ye = 0;
#pragma unroll
        for (int r = 0; r < Mc; ++r) {
          const double a = sDxi[s][r], b = sDeta[s][r];
          const int lr = t * Mc + r;
          xx += a * sx[e][lr][0]; xe += b * sx[e][lr][0];
          yx += a * sx[e][lr][1]; ye += b * sx[e][lr][1];
        }
        double xt = 0.0, yt = 0.0;
#pragma unroll
        for (int u = 0; u < Nt; ++u) {
          xt += sDtau[t][u] * sx[e][u * Mc + s][0];
          yt += sDtau[t][u] * sx[e][u * Mc + s][1];
        }
        xt *= idt;
        yt *= idt;
        const double idet = 1.0 / (xx * ye - xe * yx);
        const double xix = ye * idet, xiy = -xe * idet, etx = -yx * idet, ety = xx * idet;
        const double xit = -(xix * xt + xiy * yt), ett = -(etx * xt + ety * yt);
        double Pv[4] = {0, 0, 0, 0};
#pragma unroll
        for (int r = 0; r < Mc; ++r) {
          const double a = sDxi[s][r], b = sDeta[s][r];
          const double wx = a * xix + b * etx, wy = a * xiy + b * ety, wt = a * xit + b * ett;
          const int lr = t * Mc + r;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            Pv[v] += wx * sf[e][lr][v];
            Pv[v] += wy * sg[e][lr][v];
            Pv[v] += wt * sq[e][lr][v];
          }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) sP[e][l][v] = -Pv[v];
      } else if (full) {  // tau = 0 node, first iteration: P (eq. pdef, eq. Jac) keeping its parts
        double Qx[4] = {0, 0, 0, 0}, Qe[4] = {0, 0, 0, 0}, fx[4] = {0, 0, 0, 0}, fe[4] = {0, 0, 0, 0};
        double gx[4] = {0, 0, 0, 0}, ge[4] = {0, 0, 0, 0};
        double xx = 0, xe = 0, yx = 0, ye = 0;
#pragma unroll
        for (int r = 0; r < Mc; ++r) {
          const double a = sDxi[s][r], b = sDeta[s][r];
          const int lr = t * Mc + r;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const double qv = sq[e][lr][v], fv = sf[e][lr][v], gv = sg[e][lr][v];
            Qx[v] += a * qv; Qe[v] += b * qv;
            fx[v] += a * fv; fe[v] += b * fv;
            gx[v] += a * gv; ge[v] += b * gv;
          }
          xx += a * sx[e][lr][0]; xe += b * sx[e][lr][0];
          yx += a * sx[e][lr][1]; ye += b * sx[e][lr][1];
        }
        double xt = 0.0, yt = 0.0;
        if (it > 0) {
#pragma unroll
          for (int u = 0; u < Nt; ++u) {
            xt += sDtau[t][u] * sx[e][u * Mc + s][0];
            yt += sDtau[t][u] * sx[e][u * Mc + s][1];
          }
          xt *= idt;
          yt *= idt;
        }
        const double idet = 1.0 / (xx * ye - xe * yx);
        const double xix = ye * idet, xiy = -xe * idet, etx = -yx * idet, ety = xx * idet;
        const double xit = -(xix * xt + xiy * yt), ett = -(etx * xt + ety * yt);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const double fs = -(fx[v] * xix + fe[v] * etx + gx[v] * xiy + ge[v] * ety);
          sP[e][l][v] = fs - (Qx[v] * xit + Qe[v] * ett);
          if (t == 0) {
            c_fs[v] = fs;
            c_Qx[v] = Qx[v];
            c_Qe[v] = Qe[v];
          }
        }
        if (t == 0) {
          c_xix = xix; c_xiy = xiy; c_etx = etx; c_ety = ety;
        }
      } else if (work && t == 0) {  // tau = 0 node after the first iteration
        double xt = 0.0, yt = 0.0;
#pragma unroll
        for (int u = 0; u < Nt; ++u) {
          xt += sDtau[0][u] * sx[e][u * Mc + s][0];
          yt += sDtau[0][u] * sx[e][u * Mc + s][1];
        }
        xt *= idt;
        yt *= idt;
        const double xit = -(c_xix * xt + c_xiy * yt), ett = -(c_etx * xt + c_ety * yt);
#pragma unroll
        for (int v = 0; v < 4; ++v) sP[e][l][v] = c_fs[v] - (c_Qx[v] * xit + c_Qe[v] * ett);
      }
      __syncthreads();
      if (work && t > 0) {  // K_tau qhat = dt M P with the tau = 0 dofs known (eqs. CGfinal, newVertPos)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          double acc = 0.0;
#pragma unroll
          for (int u = 0; u < Nt; ++u) acc += sB[t - 1][u] * sP[e][(it == 0 ? 0 : u) * Mc + s][v];
          sq[e][l][v] = sq[e][s][v] + dts * acc;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          double acc = 0.0;
#pragma unroll
          for (int u = 0; u < Nt; ++u) acc += sB[t - 1][u] * sV[e][(it == 0 ? 0 : u) * Mc + s][c];
          sx[e][l][c] = sx[e][s][c] + dts * acc;
        }
      }
      __syncthreads();
    }
    // a non-positive density or pressure at any space-time node sends the
    // element back to w_h on every time slice
    if (work) {
      const double* q = sq[e][l];
      if (!(q[0] > 0.0) || !(gm1 * (q[3] - 0.5 * (q[1] * q[1] + q[2] * q[2]) / q[0]) > 0.0)) sbad[e] = 1;
    }
    __syncthreads();
    if (work && t > 0 && sbad[e]) {
#pragma unroll
      for (int v = 0; v < 4; ++v) sq[e][l][v] = sq[e][s][v];
    }
    __syncthreads();
    if (live) {
      double* out = d.qhat + ((size_t)i * Nst + l) * 4;
#pragma unroll
      for (int v = 0; v < 4; ++v) out[v] = sq[e][l][v];
      // derived tables: edge traces and reference averages (one code path:
      // a weighted sum over each time slice's nodes, then the tau powers),
      // vertex displacements
      constexpr int nTr = 3 * Nt * 4, nItems = nTr + 4 + 6;
      for (int item = l; item < nItems; item += Nst) {
        if (item < nTr + 4) {
          const int row = item / 4, v = item % 4;  // row < 3 Nt: edge row / Nt, Gauss point row % Nt
          const double* wts = sTr[row];
          double val[Nt];
#pragma unroll
          for (int tt = 0; tt < Nt; ++tt) {
            double acc = 0.0;
#pragma unroll
            for (int r = 0; r < Mc; ++r) acc += wts[r] * sq[e][tt * Mc + r][v];
            val[tt] = acc;
          }
          double* dst = row < 3 * Nt ? d.trace + ((size_t)i * 3 * Nt + row) * Nt * 4 : d.avgc + (size_t)i * Nt * 4;
#pragma unroll
          for (int p = 0; p < Nt; ++p) {
            double acc = 0.0;
#pragma unroll
            for (int tt = 0; tt < Nt; ++tt) acc += sVt[p][tt] * val[tt];
            dst[p * 4 + v] = acc;
          }
        } else {
          const int kc = item - nTr - 4, k = kc / 2, c = kc % 2;
          const int sn = k == 0 ? 0 : (k == 1 ? M : Mc - 1);
          double vel[Nt];
#pragma unroll
          for (int tt = 0; tt < Nt; ++tt) {
            const double* q = sq[e][tt * Mc + sn];
            vel[tt] = T.eulerian ? 0.0 : q[1 + c] / q[0];
          }
          double* vd = d.vdisp + ((size_t)i * 6 + kc) * Nt;
#pragma unroll
          for (int p = 0; p < Nt; ++p) {
            double acc = 0.0;
#pragma unroll
            for (int tt = 0; tt < Nt; ++tt) acc += sVt[p][tt] * vel[tt];
            vd[p] = acc * (1.0 / (p + 1));  // p is unrolled: a constant factor
          }
        }
      }
    }
    __syncthreads();
  }
}

template <int M, int TH>
void launch_predict_t(const Tab& T, const Dev& d, int nsm, cudaStream_t s, int initial, int bpsm) {
  using S = PredShape<M, TH>;
  const int need = (d.ne + S::G - 1) / S::G;
  // sweeps: the blocks that fit on the GPU at once (the launch bounds' two or
  // three per SM), so that balanced rounds give every SM the same elements
  const int grid = initial ? need : std::min(need, nsm * (TH >= 256 ? 2 : 3));
  (void)bpsm;
  k_predict_coop<M, TH><<<grid, S::kThreads, 0, s>>>(T, d, initial, T.gts);
}

template <int M>
void launch_predict(const Tab& T, const Dev& d, int nsm, cudaStream_t s, int initial, const Tiles& tl) {
  if (tl.pred_wide) launch_predict_t<M, 256>(T, d, nsm, s, initial, tl.bpsm);
  else launch_predict_t<M, 128>(T, d, nsm, s, initial, tl.bpsm);
}

}  // namespace

void launch_plain_predict(const Tab& T, const Dev& d, int nsm, cudaStream_t s, int initial, const Tiles& tl) {
  switch (T.M) {
    case 1: launch_predict<1>(T, d, nsm, s, initial, tl); break;
    case 2: launch_predict<2>(T, d, nsm, s, initial, tl); break;
    default: launch_predict<3>(T, d, nsm, s, initial, tl); break;
  }
}

}  // namespace aw
