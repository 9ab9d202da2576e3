// Stage 4b: per-Gaussian backward of the slice, colour and projection.
//
// The blend backward leaves, for every (view, Gaussian) pair, the gradient
// of the loss with respect to that pair's record (u, v, qa, qb, qc, lo, r, g,
// b).  param_bwd_kernel runs one thread per Gaussian, loops over the cameras
// that see it and sums in registers, so no atomics are needed and each
// parameter gradient is written once:
//   geometry -- conic and 2D mean -> EWA projection -> mu_cond and
//               Sigma_cond; alpha_cond -> alpha and D (Eq. pdfv2);
//               mu_cond = mu_p + A (d - mu_d) (Eq. mu); then, once
//               per Gaussian, the Schur complement (Eq. sigma) and
//               Sigma_d^-1 back to Sigma = L L^T and the raw Cholesky,
//               opacity and mean parameters;
//   colour   -- sigmoid(sum_k beta_k Y_k(d)) (section 4.2): gradients of beta
//               and the d -> mu_p term.
// Forward quantities are recomputed from the parameters with the same
// arithmetic as the forward kernel.
//
// What bounds it: instructions at half-empty warps.  A Gaussian is seen by all
// cameras, by none or by some, as its opacity and direction have it, and a
// warp of 32 neighbours turns as often as its most visible one.  So a CTA
// takes its 128 Gaussians in the order of their number of views, which fills
// warps with equals (and lets those of unseen Gaussians go at once).  The
// parameter planes are staged in shared memory by bulk copies as in the
// projection, each thread works on its Gaussian's column, leaves its gradients
// in the same places, and the CTA writes them out plane by plane.  Against
// two kernels, geometry and colour, in Gaussian order: 146 -> 130 us at 300k /
// 8 x 800^2 (3.3 of 8 views see a Gaussian), 546 -> 456 us at 2M / 4 views
// (0.3 of 4), 1354 -> 1236 us at 500k / 64 views.
#include "common.cuh"
#include "cond.cuh"
#include "kernels.cuh"
#include "mat3.cuh"
#include "sh.cuh"
#include "stage.cuh"

namespace sixdgs {

// The camera parameters the backward reads, in shared memory with an odd
// stride in words, so that lanes at different cameras do not collide.
struct CamView {
  float r[9], t[3], campos[3], fx, fy, cx, cy, znear, limx, limy;
  float pad;
};
constexpr int kCamWords = 22;   // the leading words of a CamRec
static_assert(sizeof(CamView) == (kCamWords + 1) * 4 && (kCamWords + 1) % 2 == 1, "odd stride");

// Planes of the staged tile: mu_p, mu_d, the raw Cholesky factor, the opacity
// logit, the optional per-Gaussian lambda, then the SH coefficients.
struct BwdPlanes {
  int mu_p, mu_d, l_raw, logit, lam, sh, count;
};

__host__ __device__ inline BwdPlanes bwd_planes(int sh_degree, bool lambda) {
  BwdPlanes p;
  p.mu_p = 0;
  p.mu_d = 3;
  p.l_raw = 6;
  p.logit = 27;
  p.lam = 28;
  p.sh = p.lam + (lambda ? 1 : 0);
  p.count = p.sh + (sh_degree + 1) * (sh_degree + 1) * 3;
  return p;
}

__device__ __forceinline__ const float* bwd_src(const ProjectBwdArgs& a, const BwdPlanes& pp, int q) {
  if (q < pp.mu_d) return a.mu_p + (int64_t)q * a.n;
  if (q < pp.l_raw) return a.mu_d + (int64_t)(q - pp.mu_d) * a.n;
  if (q < pp.logit) return a.l_raw + (int64_t)(q - pp.l_raw) * a.n;
  if (q < pp.lam) return a.opacity_logit;
  if (q < pp.sh) return a.lambda_raw;
  return a.sh + (int64_t)(q - pp.sh) * a.n;
}

__device__ __forceinline__ float* bwd_dst(const ProjectBwdArgs& a, const BwdPlanes& pp, int q) {
  if (q < pp.mu_d) return a.grad_mu_p + (int64_t)q * a.n;
  if (q < pp.l_raw) return a.grad_mu_d + (int64_t)(q - pp.mu_d) * a.n;
  if (q < pp.logit) return a.grad_l_raw + (int64_t)(q - pp.l_raw) * a.n;
  if (q < pp.lam) return a.grad_opacity_logit;
  if (q < pp.sh) return a.grad_lambda_raw;   // may be null
  return a.grad_sh + (int64_t)(q - pp.sh) * a.n;
}

// Sum of a symmetric 3x3 matrix (upper triangle).
struct Sym3 {
  float m[6];
  __device__ __forceinline__ float& at(int i, int j) { return m[i == 0 ? j : i + j + 1]; }
  __device__ __forceinline__ M3 full() const {
    M3 r;
    r(0, 0) = m[0];
    r(0, 1) = r(1, 0) = m[1];
    r(0, 2) = r(2, 0) = m[2];
    r(1, 1) = m[3];
    r(1, 2) = r(2, 1) = m[4];
    r(2, 2) = m[5];
    return r;
  }
};

// The cameras that see a Gaussian (mask words of 32), ascending.
struct ViewWalk {
  const uint32_t* words;   // one every kStageTile
  uint32_t mask;
  int w, n_words;

  __device__ __forceinline__ ViewWalk(const uint32_t* words_, int n_words_)
      : words(words_), mask(n_words_ > 0 ? words_[0] : 0u), w(0), n_words(n_words_) {}
  __device__ __forceinline__ int next() {   // -1: no more
    while (mask == 0u) {
      if (++w >= n_words) return -1;
      mask = words[w * kStageTile];
    }
    const int i = __ffs(mask) - 1;
    mask &= mask - 1u;
    return w * 32 + i;
  }
};

// Geometry part for the Gaussian whose planes are at sp[q * kStageTile]: its
// gradients replace its mu_d, l_raw, logit and lambda there; gmp: its part of
// the gradient of mu_p.
__device__ __forceinline__ void geometry_bwd(const ProjectBwdArgs& a, const BwdPlanes& pp, const CamView* s_cams,
                                             float* sp, const float4* grec, ViewWalk walk, float* gmp) {
  const int64_t n = a.n;
  float mp[3], md[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    mp[i] = sp[(pp.mu_p + i) * kStageTile];
    md[i] = sp[(pp.mu_d + i) * kStageTile];
  }
  const float lam = a.lambda_raw ? sigmoidf_(sp[pp.lam * kStageTile]) : a.lambda_opa;
  CondState cs;
  const bool ok = condition_from([&](int q) { return sp[(pp.l_raw + q) * kStageTile]; }, sp[pp.logit * kStageTile], cs);
  const M3 &A = cs.A, &S = cs.Sdi, &Sc = cs.Sc;
  const float alpha = cs.alpha;

  M3 gA = zero3();
  Sym3 gS = {}, gSc = {};
  float gmd[3] = {0.f, 0.f, 0.f}, galpha = 0.f, glam = 0.f;

  // the next camera's record gradients are loaded a turn ahead
  int v_next = ok ? walk.next() : -1;
  float4 ga_next, gb_next;
  if (v_next >= 0) {
    ga_next = grec[(int64_t)v_next * n * 3];
    gb_next = grec[(int64_t)v_next * n * 3 + 1];
  }
  while (v_next >= 0) {
    const CamView& cam = s_cams[v_next];
    const float4 ga = ga_next, gb = gb_next;
    v_next = walk.next();
    if (v_next >= 0) {
      ga_next = grec[(int64_t)v_next * n * 3];
      gb_next = grec[(int64_t)v_next * n * 3 + 1];
    }
    // ---- forward recomputation (same arithmetic as project_fwd_kernel) ----
    float dv[3] = {mp[0] - cam.campos[0], mp[1] - cam.campos[1], mp[2] - cam.campos[2]};
    const float inv_len = rsqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
    const float d[3] = {dv[0] * inv_len, dv[1] * inv_len, dv[2] * inv_len};
    const float delta[3] = {d[0] - md[0], d[1] - md[1], d[2] - md[2]};
    float Ad[3], Sdl[3];
    mat_vec(A, delta, Ad);
    mat_vec(S, delta, Sdl);
    const float mc[3] = {mp[0] + Ad[0], mp[1] + Ad[1], mp[2] + Ad[2]};
    const float D = delta[0] * Sdl[0] + delta[1] * Sdl[1] + delta[2] * Sdl[2];
    const float f = __expf(-lam * D);
    const float alpha_cond = alpha * f;
    float t[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      t[i] = cam.r[i * 3] * mc[0] + cam.r[i * 3 + 1] * mc[1] + cam.r[i * 3 + 2] * mc[2] + cam.t[i];
    const float iz = 1.f / t[2];
    const float rx_raw = t[0] * iz, ry_raw = t[1] * iz;
    const float rx = fminf(cam.limx, fmaxf(-cam.limx, rx_raw));
    const float ry = fminf(cam.limy, fmaxf(-cam.limy, ry_raw));
    const float j00 = cam.fx * iz, j02 = -cam.fx * rx * iz;
    const float j11 = cam.fy * iz, j12 = -cam.fy * ry * iz;
    float T0[3], T1[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      T0[j] = j00 * cam.r[j] + j02 * cam.r[6 + j];
      T1[j] = j11 * cam.r[3 + j] + j12 * cam.r[6 + j];
    }
    float U0[3], U1[3];
    mat_t_vec(Sc, T0, U0);
    mat_t_vec(Sc, T1, U1);
    const float ca = U0[0] * T0[0] + U0[1] * T0[1] + U0[2] * T0[2] + kDilation;
    const float cb = U0[0] * T1[0] + U0[1] * T1[1] + U0[2] * T1[2];
    const float cc = U1[0] * T1[0] + U1[1] * T1[1] + U1[2] * T1[2] + kDilation;
    const float det = ca * cc - cb * cb;
    const float idet = 1.f / det;
    const float idet2 = idet * idet;
    // ---- record gradients -> conic and alpha_cond ----
    // The blend leaves the moments M = sum over pixels of g, g dx, g dy,
    // g dx^2, g dx dy, g dy^2 with g = (dL/dq) / ln 2 and
    // q = qa dx^2 + qb dx dy + qc dy^2 + lo, dx = u - px, dy = v - py.
    const float con_a0 = cc * idet, con_b0 = -cb * idet, con_c0 = ca * idet;
    const float qa = -0.5f * kLog2e * con_a0, qb = -kLog2e * con_b0, qc = -0.5f * kLog2e * con_c0;
    const float du = kLn2 * (2.f * qa * ga.x + qb * ga.y);
    const float dvv = kLn2 * (qb * ga.x + 2.f * qc * ga.y);
    const float dcon_a = -0.5f * kLog2e * kLn2 * ga.z;   // dq/dcon_a = -1/2 log2(e) dx^2
    const float dcon_b = -kLog2e * kLn2 * ga.w;
    const float dcon_c = -0.5f * kLog2e * kLn2 * gb.x;
    const float dalpha_cond = gb.y / alpha_cond;         // lo = log2(alpha_cond): ln 2 cancels
    // conic = (cc, -cb, ca) / det  ->  (ca, cb, cc)
    const float d_ca = (-dcon_a * cc * cc + dcon_b * cb * cc - dcon_c * cb * cb) * idet2;
    const float d_cb = (2.f * dcon_a * cb * cc - dcon_b * (det + 2.f * cb * cb) + 2.f * dcon_c * ca * cb) * idet2;
    const float d_cc = (-dcon_a * cb * cb + dcon_b * ca * cb - dcon_c * ca * ca) * idet2;
    // (ca, cb, cc) = (T0 Sc T0, T0 Sc T1, T1 Sc T1) (+ dilation)
    // (the symmetric part of dL/dSigma_cond, which is all that reaches Sigma)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j)
        gSc.at(i, j) += d_ca * T0[i] * T0[j] + 0.5f * d_cb * (T0[i] * T1[j] + T1[i] * T0[j]) + d_cc * T1[i] * T1[j];
    float dT0[3], dT1[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      dT0[j] = 2.f * d_ca * U0[j] + d_cb * U1[j];
      dT1[j] = d_cb * U0[j] + 2.f * d_cc * U1[j];
    }
    // T = J R
    const float dj00 = dT0[0] * cam.r[0] + dT0[1] * cam.r[1] + dT0[2] * cam.r[2];
    const float dj02 = dT0[0] * cam.r[6] + dT0[1] * cam.r[7] + dT0[2] * cam.r[8];
    const float dj11 = dT1[0] * cam.r[3] + dT1[1] * cam.r[4] + dT1[2] * cam.r[5];
    const float dj12 = dT1[0] * cam.r[6] + dT1[1] * cam.r[7] + dT1[2] * cam.r[8];
    float dtx = 0.f, dty = 0.f, dtz = 0.f;
    dtz += -j00 * iz * dj00 - j11 * iz * dj11;
    dtz += -j02 * iz * dj02 - j12 * iz * dj12;   // at fixed rx, ry
    const float drx = -cam.fx * iz * dj02, dry = -cam.fy * iz * dj12;
    if (fabsf(rx_raw) <= cam.limx) {
      dtx += drx * iz;
      dtz += -drx * t[0] * iz * iz;
    }
    if (fabsf(ry_raw) <= cam.limy) {
      dty += dry * iz;
      dtz += -dry * t[1] * iz * iz;
    }
    // 2D mean
    dtx += du * cam.fx * iz;
    dty += dvv * cam.fy * iz;
    dtz += -(du * cam.fx * t[0] + dvv * cam.fy * t[1]) * iz * iz;
    // t = R mu_cond + t_w
    float dmc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) dmc[i] = cam.r[i] * dtx + cam.r[3 + i] * dty + cam.r[6 + i] * dtz;
    // ---- slice backward (Eq. mu, Eq. pdfv2, Eq. alpha) ----
    float ddelta[3];
    mat_t_vec(A, dmc, ddelta);
    const float dD = -lam * alpha_cond * dalpha_cond;
    galpha += f * dalpha_cond;
    glam -= D * alpha_cond * dalpha_cond;   // d alpha_cond / d lambda = -D alpha_cond
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gmp[i] += dmc[i];
      ddelta[i] += 2.f * dD * Sdl[i];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        gA(i, j) += dmc[i] * delta[j];
        if (j >= i) gS.at(i, j) += dD * delta[i] * delta[j];
      }
    }
    const float dot = d[0] * ddelta[0] + d[1] * ddelta[1] + d[2] * ddelta[2];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gmd[i] -= ddelta[i];
      gmp[i] += (ddelta[i] - d[i] * dot) * inv_len;
    }
  }

  // L and the Sigma blocks again (cheaper than keeping them over the loop)
  float L[6][6];
  cholesky_from([&](int q) { return sp[(pp.l_raw + q) * kStageTile]; }, L);
  M3 Sp, P, Sd;
  sigma_blocks(L, Sp, P, Sd);
  // ---- Schur complement and inverse (Eq. sigma) back to Sigma blocks ----
  // Sc = Sp - A P^T, A = P S, S = Sd^-1
  const M3 gScm = gSc.full();
  const M3 GA = sub(gA, mul(gScm, P));
  const M3 GP = sub(mul(GA, S), mul(gScm, A));   // G_A S - gSc^T A
  const M3 GS = add(mul_at(P, GA), gS.full());
  const M3 GSd = mul(mul(S, GS), S);   // dL/dSd = -S GS S (sign applied below)
  // ---- Sigma = L L^T back to L ----
  float dL[6][6];
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) dL[i][j] = 0.f;
  // symmetric parts
  M3 Gp2, Gd2;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Gp2(i, j) = 2.f * gScm(i, j);
      Gd2(i, j) = -(GSd(i, j) + GSd(j, i));
    }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float lpp = 0.f, ldp = 0.f, ldd = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        lpp += Gp2(i, k) * L[k][j] + GP(i, k) * L[3 + k][j];  // ((G+G^T) Lpp + G_P Ldp)_{ij}
        ldp += GP(k, i) * L[k][j] + Gd2(i, k) * L[3 + k][j];  // (G_P^T Lpp + (Gd+Gd^T) Ldp)_{ij}
        ldd += Gd2(i, k) * L[3 + k][3 + j];                   // ((Gd+Gd^T) Ldd)_{ij}
      }
      dL[i][j] = lpp;
      dL[3 + i][j] = ldp;
      dL[3 + i][3 + j] = ldd;
    }
  int k = 6;
#pragma unroll
  for (int i = 0; i < 6; ++i) sp[(pp.l_raw + i) * kStageTile] = ok ? dL[i][i] * L[i][i] : 0.f;
#pragma unroll
  for (int i = 1; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j) {
      const float v = L[i][j];
      sp[(pp.l_raw + k++) * kStageTile] = ok ? dL[i][j] * 0.5f * (1.f - v * v) : 0.f;
    }
  sp[pp.logit * kStageTile] = ok ? galpha * alpha * (1.f - alpha) : 0.f;
  if (a.lambda_raw) sp[pp.lam * kStageTile] = ok ? glam * lam * (1.f - lam) : 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) sp[(pp.mu_d + i) * kStageTile] = gmd[i];
}

// Colour part: the gradients replace the Gaussian's SH planes and mu_p (with
// the geometry part gmp added).
__device__ __forceinline__ void colour_bwd(const ProjectBwdArgs& a, const BwdPlanes& pp, const CamView* s_cams,
                                           float* sp, const float4* grec, const float4* rec, ViewWalk walk,
                                           const float* gmp) {
  const int64_t n = a.n;
  const int K = (a.sh_degree + 1) * (a.sh_degree + 1);
  const float mp[3] = {sp[pp.mu_p * kStageTile], sp[(pp.mu_p + 1) * kStageTile], sp[(pp.mu_p + 2) * kStageTile]};
  float* sh = sp + pp.sh * kStageTile;
  float dbeta[kMaxShCoeffs][3];
#pragma unroll
  for (int k = 0; k < kMaxShCoeffs; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) dbeta[k][c] = 0.f;
  float dmp[3] = {0.f, 0.f, 0.f};
  // the next camera's colour gradients and colour are loaded a turn ahead
  int v_next = walk.next();
  float4 gb_next, rb_next;
  float gz_next = 0.f, rz_next = 0.f;
  auto fetch = [&]() {
    const int64_t p = (int64_t)v_next * n * 3;
    gb_next = grec[p + 1];
    gz_next = grec[p + 2].x;
    rb_next = rec[p + 1];
    rz_next = rec[p + 2].x;
  };
  if (v_next >= 0) fetch();
  while (v_next >= 0) {
    const CamView& cam = s_cams[v_next];
    const float drgb[3] = {gb_next.z, gb_next.w, gz_next};
    const float rgb[3] = {rb_next.z, rb_next.w, rz_next};
    v_next = walk.next();
    if (v_next >= 0) fetch();
    if (drgb[0] == 0.f && drgb[1] == 0.f && drgb[2] == 0.f) continue;
    float dv[3] = {mp[0] - cam.campos[0], mp[1] - cam.campos[1], mp[2] - cam.campos[2]};
    const float inv_len = rsqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
    const float d[3] = {dv[0] * inv_len, dv[1] * inv_len, dv[2] * inv_len};
    float dpre[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) dpre[c] = drgb[c] * rgb[c] * (1.f - rgb[c]);
    float Y[kMaxShCoeffs], w[kMaxShCoeffs];
#pragma unroll
    for (int k = 0; k < kMaxShCoeffs; ++k) Y[k] = 0.f;
    sh_basis(a.sh_degree, d[0], d[1], d[2], Y);
#pragma unroll
    for (int k = 0; k < kMaxShCoeffs; ++k) {
      w[k] = 0.f;
      if (k < K) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          dbeta[k][c] += dpre[c] * Y[k];
          w[k] += dpre[c] * sh[(k * 3 + c) * kStageTile];
        }
      }
    }
    float gd[3];
    sh_grad(a.sh_degree, d[0], d[1], d[2], w, gd);
    // d = v / |v|: dv = (gd - d (d . gd)) / |v|
    const float dot = d[0] * gd[0] + d[1] * gd[1] + d[2] * gd[2];
#pragma unroll
    for (int i = 0; i < 3; ++i) dmp[i] += (gd[i] - d[i] * dot) * inv_len;
  }
#pragma unroll
  for (int k = 0; k < kMaxShCoeffs; ++k)
    if (k < K)
#pragma unroll
      for (int c = 0; c < 3; ++c) sh[(k * 3 + c) * kStageTile] = dbeta[k][c];
#pragma unroll
  for (int i = 0; i < 3; ++i) sp[(pp.mu_p + i) * kStageTile] = dmp[i] + gmp[i];
}

constexpr int kBins = 288;   // numbers of views, 0 to 256, and some

// 4 CTAs per SM (128 registers; 5 at 102 registers spill: 204 instead of 131 us).
__global__ void __launch_bounds__(kStageTile, 4) param_bwd_kernel(ProjectBwdArgs a) {
  after_previous();
  extern __shared__ float4 s_dyn[];
  __shared__ uint64_t s_bars[2];
  __shared__ uint32_t s_bin[kBins];   // Gaussians of every number of views
  __shared__ uint8_t s_order[kStageTile];
  const BwdPlanes pp = bwd_planes(a.sh_degree, a.lambda_raw != nullptr);
  float* tile = reinterpret_cast<float*>(s_dyn);
  const int n_words = (a.n_cams + 31) / 32;
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(tile + pp.count * kStageTile);
  CamView* s_cams = reinterpret_cast<CamView*>(s_mask + n_words * kStageTile);
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t n = a.n, g0 = (int64_t)blockIdx.x * kStageTile;
  const int m = (int)min((int64_t)kStageTile, n - g0);
  const bool bulk = a.bulk != 0;
  for (int i = tid; i < kBins; i += kStageTile) s_bin[i] = 0u;
  {
    const float* src = reinterpret_cast<const float*>(a.cams);
    float* dst = reinterpret_cast<float*>(s_cams);
    for (int i = tid; i < a.n_cams * kCamWords; i += kStageTile) {
      const int v = i / kCamWords, w = i - v * kCamWords;
      dst[v * (kCamWords + 1) + w] = src[v * (int)(sizeof(CamRec) / 4) + w];
    }
  }
  stage_issue(tile, pp.count, pp.sh, [&](int q) { return bwd_src(a, pp, q); }, g0, m, bulk, s_bars);

  // the views of every Gaussian, and the Gaussians by falling number of views
  uint32_t views = 0, rank = 0;
  if (tid < m) {
    for (int w = 0; w < n_words; ++w) {
      const uint32_t* nt = a.ntiles + (int64_t)(w * 32) * n + g0 + tid;
      const int c = min(32, a.n_cams - w * 32);
      uint32_t mask = 0u;
#pragma unroll 8
      for (int i = 0; i < c; ++i) mask |= (nt[(int64_t)i * n] != 0u ? 1u : 0u) << i;
      s_mask[w * kStageTile + tid] = mask;
      views += __popc(mask);
    }
    rank = atomicAdd(&s_bin[views], 1u);
  }
  __syncthreads();
  if (tid < 32) {   // Gaussians with more views: a suffix sum over the bins, 9 a lane
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < kBins / 32; ++i) sum += s_bin[lane * (kBins / 32) + i];
    uint32_t above = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_down_sync(0xffffffffu, above, o);
      if (lane + o < 32) above += y;
    }
    above -= sum;
#pragma unroll
    for (int i = kBins / 32 - 1; i >= 0; --i) {
      const uint32_t c = s_bin[lane * (kBins / 32) + i];
      s_bin[lane * (kBins / 32) + i] = above;
      above += c;
    }
  }
  __syncthreads();
  const uint32_t seen = s_bin[0];   // those with more than no views come first
  if (tid < m) s_order[s_bin[views] + rank] = (uint8_t)tid;
  __syncthreads();

  if (!stage_wait(s_bars, 0, bulk, a.spin_budget)) raise_status(a.status, SIXDGS_ERR_TIMEOUT);
  if (!stage_wait(s_bars, 1, bulk, a.spin_budget)) raise_status(a.status, SIXDGS_ERR_TIMEOUT);
  if (tid < m) {
    const int gl = s_order[tid];
    float* sp = tile + gl;
    if ((uint32_t)tid < seen) {
      const ViewWalk walk(s_mask + gl, n_words);
      const float4* grec = reinterpret_cast<const float4*>(a.grad_rec) + (g0 + gl) * 3;
      const float4* rec = reinterpret_cast<const float4*>(a.rec) + (g0 + gl) * 3;
      float gmp[3] = {0.f, 0.f, 0.f};
      geometry_bwd(a, pp, s_cams, sp, grec, walk, gmp);
      colour_bwd(a, pp, s_cams, sp, grec, rec, walk, gmp);
    } else {
      for (int q = 0; q < pp.count; ++q) sp[q * kStageTile] = 0.f;
    }
  }
  __syncthreads();

  // the gradients, a warp per plane
  const bool acc = a.accumulate != 0;
  for (int q = tid >> 5; q < pp.count; q += kStageTile / 32) {
    float* dst = bwd_dst(a, pp, q);
    if (!dst) continue;
    dst += g0;
    const float* src = tile + q * kStageTile;
    if (m == kStageTile && !acc && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
      reinterpret_cast<float4*>(dst)[lane] = reinterpret_cast<const float4*>(src)[lane];
    } else {
      for (int i = lane; i < m; i += 32) dst[i] = acc ? dst[i] + src[i] : src[i];
    }
  }
}

void launch_param_bwd(const ProjectBwdArgs& a, cudaStream_t stream) {
  if (a.n == 0) return;
  const BwdPlanes pp = bwd_planes(a.sh_degree, a.lambda_raw != nullptr);
  const size_t smem = (size_t)pp.count * kStageTile * 4 + (size_t)((a.n_cams + 31) / 32) * kStageTile * 4 +
                      sizeof(CamView) * (size_t)a.n_cams;
  if (smem > 40 * 1024)
    cudaFuncSetAttribute(param_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_after(param_bwd_kernel, (unsigned)((a.n + kStageTile - 1) / kStageTile), kStageTile, smem, 1, stream, a);
}

}  // namespace sixdgs
