// FP32 operator of the mixed cycle in edge form (Eq. 2.3 with the element
// matrices of Eq. 3.5; on coarse levels the heterogeneous operator of Eq.
// 2.9), fused with the smoother and residual epilogues: every FP32 level of
// more than kPointMaxN cubes per axis.
//
// The fluxes along the grid's axis edges and their weights are those of
// stencil_edge.cu, with the weights formed from the element coefficients here
// (six values per cube; a record of 27 per vertex would double the traffic
// of an operator that HBM should bound).
//
// What bounds it: HBM for the smoothing steps, instruction issue for the
// residual.  60 to 96 bytes a vertex at the copy rate leave an SM 90 to 140
// cycles for each 32 vertices; the per-cube kernel this replaces issued 533
// instructions a vertex, this one about 320.
// Measured at 256^3 cubes (per-cube kernel -> this; in brackets the method's
// bytes over the time, of the measured copy rate): residual 368 -> 216 us (0.69),
// first step 392 -> 251 us (0.72), later step with FP64 result 414 -> 325 us
// (0.74), step from zero 444 -> 251 us (0.60; 0.72 with its first iterate, which
// the producer of b writes in 36 us); at 128^3 cubes 66-82 -> 34-46 us.
//
// Tiling: a CTA owns 32 x 16 vertex columns starting at vertex (1, 1) and
// marches a chunk of z-planes; n a multiple of 32 then wastes no lane.  Eight
// warps hold two consecutive rows per thread, so that of the ten
// vertices a pair needs on each plane most are read once, and the y flux
// between the rows stays in registers.  The fluxes that enter the tile (x
// edges left of it, y edges below it), the halo copies and the Dirichlet
// entries of column 0 and row 0 are spread over the warps.  Vectors and
// coefficients are staged by cp.async two planes ahead.  Two barriers per
// plane: staged data visible; y and left x fluxes exchanged.
//
// Every flux is formed with the same operations wherever it is computed, and
// every vertex adds its six in one fixed order: results depend on no tile
// position and no z-chunk, and the batched form gives the same bits.
#include <algorithm>

#include "agca_internal.cuh"
#include "device_ops.cuh"

namespace agca {

namespace {

constexpr int FX = 32, FR = 2, FW = 8, FY = FR * FW;  // owned columns, rows per thread, warps, owned rows
constexpr int FNT = 32 * FW;
constexpr int VW = FX + 2, VT = VW * (FY + 2);        // vertex tile: columns -1 .. 32, rows -1 .. 16
constexpr int CP = 200, CT = CP * (FY + 1);           // cube tile: 6 x (columns -1 .. 31) floats a row, rows -1 .. 15
constexpr int CQ = CP / 4 * (FY + 1);                 // 16-byte pieces of a cube layer
constexpr int HV = 2 * (FY + 2) + 2 * FX;             // halo vertices
constexpr int CRING = 3;                              // cube layers k - 1 .. k + 1
constexpr int kHaloWarp = 1, kLeftWarp = FW - 1;      // first warp copying halo vertices; warp of the left fluxes
static_assert(HV <= 32 * (kLeftWarp - kHaloWarp), "one halo entry per thread");
static_assert(CP >= 6 * (FX + 1) && CP % 4 == 0, "a cube row in 16-byte pieces");

constexpr int NS = 3;                                 // vertex ring: planes k .. k + 2
// epilogue vectors staged by their own thread a plane ahead: b and D^-1 (the
// previous iterate uses plain loads: with more than about 97 KB a block, two
// blocks leave too little L1 for the copies in flight)
template <int MODE>
__host__ __device__ constexpr int f32_fields() {
  return MODE == ST_APPLY ? 0 : (MODE == ST_RESID ? 1 : 2);
}
// shared memory in bytes: coefficient ring [CRING][CT], vertex ring
// [NS][3][VT], epilogue vectors [2][3 fields][FX * FY], exchanged fluxes
template <int MODE>
__host__ __device__ constexpr size_t f32_smem() {
  return 4 * ((size_t)CRING * CT + (size_t)NS * 3 * VT + (size_t)2 * 3 * f32_fields<MODE>() * FX * FY +
              (size_t)3 * (FW + 1) * 32 + (size_t)3 * FY);
}

// cp.async of 4 bytes from base + off (bytes), zero fill where !ok
__device__ __forceinline__ void cpa4(unsigned dst, const void* base, unsigned off, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst),
               "l"(static_cast<const char*>(base) + off), "r"(ok ? 4 : 0)
               : "memory");
}
// 16 bytes past L1
__device__ __forceinline__ void cpa16(unsigned dst, const void* base, unsigned off) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(static_cast<const char*>(base) + off)
               : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cpa_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// an off-axis flux component: H d plus the four weighted differences
__device__ __forceinline__ float flux(float hd, float da, float w0, float db, float w1, float dc, float w2, float dd,
                                      float w3) {
  return fmaf(dd, w3, fmaf(dc, w2, fmaf(db, w1, fmaf(da, w0, hd))));
}

// One staged vertex: byte offset off of its component 0, shared address d of its entry
__device__ __forceinline__ void stage_vertex(const float* x, unsigned d, unsigned off, bool ok, int V) {
  off = ok ? off : 0u;
#pragma unroll
  for (int c = 0; c < 3; ++c) cpa4(d + 4 * c * VT, x + c * V, off, ok);
}

struct V3 {
  float x, y, z;
};
__device__ __forceinline__ V3 ld3(const float* p) { return V3{p[0], p[VT], p[2 * VT]}; }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }

template <int MODE, bool STEN, bool WIDE>
__device__ __forceinline__ void f32_block(const LevelOp<float>& op, const StencilArgs<float>& a, const int zch,
                                          const int bx, const int by, const int bz, float* sm) {
  constexpr int NF = f32_fields<MODE>();
  const int n = op.n, nv = n + 1, plane = nv * nv, V = plane * nv, n2 = n * n;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = 1 + bx * FX, y0 = 1 + by * FY;
  const int za = 1 + bz * zch, zb = min(za + zch, n + 1);
  float* cf = sm;                               // [CRING][FY + 1][CP]
  float* xs = cf + CRING * CT;                  // [NS][3][VT]
  float* es = xs + NS * 3 * VT;                     // [2][NF * 3][FNT * FR]: epilogue vectors
  float* fy = es + 2 * 3 * NF * FX * FY;        // [FW + 1][3][32]: y fluxes entering warp w's first row
  float* fxl = fy + 3 * (FW + 1) * 32;          // [3][FY]: x fluxes entering column 0

  const int col = x0 + lane, row = y0 + FR * w;
  const int ev = (FR * w + 1) * VW + lane + 1;  // tile index of the first row's vertex
  const int ec = (FR * w + 1) * CP + 6 * (lane + 1);  // and of its cube
  const bool ok0 = col < n && row < n, ok1 = col < n && row + 1 < n;  // interior in the plane (col, row >= 1)
  const int gv = col + nv * row;
  // this thread's halo vertex (warps 1 .. 4)
  int he = -1, hg = 0;
  bool hok = false;
  {
    const int q = (int)threadIdx.x - 32 * kHaloWarp;
    if (q >= 0 && q < HV) {
      constexpr int S = FY + 2;
      const int lx = q < S ? -1 : (q < 2 * S ? FX : (q < 2 * S + FX ? q - 2 * S : q - 2 * S - FX));
      const int ly = q < S ? q - 1 : (q < 2 * S ? q - S - 1 : (q < 2 * S + FX ? -1 : FY));
      he = (ly + 1) * VW + lx + 1;
      hg = x0 + lx + nv * (y0 + ly);
      hok = x0 + lx > 0 && y0 + ly > 0 && x0 + lx < n && y0 + ly < n;
    }
  }
  // this thread's pieces of a cube layer: the rows start at column x0 - 1, a
  // multiple of 32, and n is even, so they are 16-byte aligned.  A piece that
  // begins beyond the last column or row is not copied: those cubes enter
  // only Dirichlet outputs.  (A piece that begins within a row ends within it: a
  // row holds 6 (n - x0 + 1) values from its start, a multiple of four.)
  unsigned cg[(CQ + FNT - 1) / FNT];
#pragma unroll
  for (int i = 0; i < (CQ + FNT - 1) / FNT; ++i) {
    const int q = (int)threadIdx.x + FNT * i, r = q / (CP / 4), p = q - r * (CP / 4);
    const int cr = y0 - 1 + r;
    const bool use = q < CQ && cr < n && 4 * p < 6 * (n - (x0 - 1)) && 4 * p < 6 * (FX + 1);
    cg[i] = use ? 24u * (unsigned)(x0 - 1 + n * cr) + 16u * p : ~0u;
  }

  // Dirichlet entries of column 0 and row 0: one per thread of warps 2, 3 and 4
  int ze = -1;
  if (bx == 0 && w == 2 && lane < FY && y0 + lane <= n) ze = nv * (y0 + lane);
  if (by == 0 && w == 3 && col <= n) ze = col;
  if (bx == 0 && by == 0 && w == 4 && lane == 0) ze = 0;

  const unsigned cf_s = (unsigned)__cvta_generic_to_shared(cf), xs_s = (unsigned)__cvta_generic_to_shared(xs);
  const unsigned es_s = (unsigned)__cvta_generic_to_shared(es);
  // plane p into ring slot sx
  auto stage_plane = [&](int p, int sx) {
    const bool zin = p > 0 && p < n;
    const unsigned d = xs_s + sx * (4 * 3 * VT), o = 4u * (unsigned)(p * plane);
    stage_vertex(a.x, d + 4 * ev, o + 4u * gv, ok0 && zin, V);
    stage_vertex(a.x, d + 4 * (ev + VW), o + 4u * (gv + nv), ok1 && zin, V);
    if (he >= 0) stage_vertex(a.x, d + 4 * he, o + 4u * hg, hok && zin, V);
  };
  auto stage_layer = [&](int kc, int sc) {
    if (kc >= n) return;  // enters only the Dirichlet plane n
    const unsigned d = cf_s + sc * (4 * CT) + 16 * threadIdx.x, o = 24u * (unsigned)(kc * n2);
#pragma unroll
    for (int i = 0; i < (CQ + FNT - 1) / FNT; ++i)
      if (cg[i] != ~0u) cpa16(d + 16 * FNT * i, op.coef, o + cg[i]);
  };
  // epilogue vectors of plane p into slot p & 1
  auto stage_epilogue = [&](int p) {
    if (NF == 0) return;
    const bool zin = p > 0 && p < n;
    const unsigned d = es_s + (p & 1) * (4 * 3 * NF * FX * FY) + 4 * threadIdx.x;
#pragma unroll
    for (int r = 0; r < FR; ++r) {
      const bool ok = (r ? ok1 : ok0) && zin;
      const unsigned o = ok ? 4u * (unsigned)(gv + r * nv + p * plane) : 0u;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const unsigned e = d + 4 * FNT * r + 4 * FX * FY * c;
        cpa4(e, a.b + c * V, o, ok);
        if (NF > 1) cpa4(e + 4 * 3 * FX * FY, a.invD + c * V, o, ok);
      }
    }
  };
  auto put = [&](int v, int c, float o) {
    if (WIDE)
      (a.out64 + c * (int64_t)V)[(unsigned)v] = (double)o;  // the mixed cycle's result, widened
    else
      (a.out + c * V)[(unsigned)v] = o;
  };
  // halo plane za - 1 and plane za, layer za - 1
  stage_plane(za - 1, 0);
  stage_plane(za, 1);
  stage_layer(za - 1, 0);
  cpa_commit();

  V3 A[2][FR + 1], B[2][FR + 1];        // columns lane, lane + 1; rows 0 .. 2; planes k and k + 1
  float mx[FR + 1], my[FR], ml[FR];     // plane k - 1: x of rows -1 .. 1, y of rows 0, 1, y of column lane - 1
  float by_ = 0.f, bl_ = 0.f;           // warp 0, plane k - 1: y of row -1, columns lane and lane - 1
  float lx0 = 0.f, lx1 = 0.f;           // left fluxes, plane k - 1: x of column -1, rows j - 1 and j
  float fz[FR][3];                      // flux of the z edge below
#pragma unroll
  for (int r = 0; r < FR; ++r) my[r] = ml[r] = fz[r][0] = fz[r][1] = fz[r][2] = 0.f;
#pragma unroll
  for (int r = 0; r <= FR; ++r) mx[r] = 0.f;

  int s0 = 0, c0 = 0;  // slots of vertex plane k and of cube layer k
  auto layer = [&](const int k, V3(&Pa)[FR + 1], V3(&Pb)[FR + 1], V3(&Na)[FR + 1], V3(&Nb)[FR + 1]) {
    const bool full = k >= za;  // the halo plane supplies only its z fluxes
    const int s1 = s0 + 1 == NS ? 0 : s0 + 1, s2 = s1 + 1 == NS ? 0 : s1 + 1;
    const int c1 = c0 == 2 ? 0 : c0 + 1, cm = c1 == 2 ? 0 : c1 + 1;
    cpa_wait0();
    __syncthreads();  // plane k + 1 and cube layer k staged; slots of plane k - 1 and layer k - 2 free
    if (k + 1 < zb) {
      stage_plane(k + 2, s2);
      stage_layer(k + 1, c1);
      stage_epilogue(k + 1);
    }
    cpa_commit();
    const float* xn = xs + s1 * 3 * VT + ev;
    const float* xp = xs + s0 * 3 * VT + ev;
    const float* q = cf + c0 * CT + ec;                              // layer k
    const float* qm = cf + cm * CT + ec;                             // layer k - 1
    if (!full) {
#pragma unroll
      for (int r = 0; r <= FR; ++r) {
        Pa[r] = ld3(xp + r * VW);
        Pb[r] = ld3(xp + r * VW + 1);
      }
    }
#pragma unroll
    for (int r = 0; r <= FR; ++r) {
      Na[r] = ld3(xn + r * VW);
      Nb[r] = ld3(xn + r * VW + 1);
    }
    const bool zin = k > 0 && k < n;
    float F[FR][3][3];  // [row][edge axis][component]
    V3 am1 = ld3(xp - VW);            // row r - 1
    V3 lm = ld3(xp - VW - 1);         // row r - 1, column lane - 1
    // layer k: row r - 1 types 2, 3, 5; both - 1 types 0, 2
    float2 d23 = ld2(q - CP + 2);
    float dxy0 = q[-CP - 6], dxy2 = q[-CP - 6 + 2];
    // layer k - 1: row r - 1 types 3, 5
    float y3 = qm[-CP + 3], y5 = qm[-CP + 5];
    if (w == 0 && full) {  // y edge from row -1 into row 0
      const float v2 = d23.x, v3 = d23.y, x1 = qm[-CP - 6 + 1], x4 = qm[-CP - 6 + 4];
      const float h = ((v2 + v3) + (dxy0 + y5)) + (x1 + x4);
      const float hd = h * (Pa[0].y - am1.y);
      fy[lane] = flux(h * (Pa[0].x - am1.x), Pb[0].y - Pa[0].y, v2 + y5, am1.y - lm.y, dxy0 + x4, Nb[0].y - Na[0].y, v3,
                      by_ - bl_, x1);
      fy[32 + lane] = hd + hd;
      fy[64 + lane] = flux(h * (Pa[0].z - am1.z), Na[0].y - Pa[0].y, v3 + dxy0, am1.y - by_, y5 + x1,
                           Nb[0].y - Pb[0].y, v2, lm.y - bl_, x4);
    }
    by_ = am1.y;
    bl_ = lm.y;
    const float mx_next = am1.x;
#pragma unroll
    for (int r = 0; r < FR; ++r) {
      const V3 a0 = Pa[r], a1 = Pa[r + 1], b0 = Pb[r], b1 = Pb[r + 1];
      const V3 na0 = Na[r], na1 = Na[r + 1], nb0 = Nb[r], nb1 = Nb[r + 1];
      const V3 l0 = ld3(xp + r * VW - 1);
      const float2 v01 = ld2(q + r * CP), v23 = ld2(q + r * CP + 2), v45 = ld2(q + r * CP + 4);
      const float2 x01 = ld2(q + r * CP - 6);             // column - 1, layer k
      const float2 m45 = ld2(qm + r * CP + 4);              // own, layer k - 1
      const float x1 = qm[r * CP - 6 + 1], x4 = qm[r * CP - 6 + 4];  // column - 1, layer k - 1
      if (full) {
        {  // x edge
          const float h = ((v01.x + v01.y) + (d23.x + m45.x)) + (y3 + y5);
          const float hd = h * (b0.x - a0.x);
          F[r][0][0] = hd + hd;
          F[r][0][1] = flux(h * (b0.y - a0.y), b1.x - b0.x, v01.x + m45.x, a0.x - am1.x, d23.x + y5, nb1.x - nb0.x,
                            v01.y, mx[r + 1] - mx[r], y3);
          F[r][0][2] = flux(h * (b0.z - a0.z), nb0.x - b0.x, v01.y + d23.x, a0.x - mx[r + 1], m45.x + y3,
                            nb1.x - b1.x, v01.x, am1.x - mx[r], y5);
        }
        {  // y edge
          const float h = ((v23.x + v23.y) + (x01.x + m45.y)) + (x1 + x4);
          const float hd = h * (a1.y - a0.y);
          F[r][1][1] = hd + hd;
          F[r][1][0] = flux(h * (a1.x - a0.x), b1.y - a1.y, v23.x + m45.y, a0.y - l0.y, x01.x + x4, nb1.y - na1.y,
                            v23.y, my[r] - ml[r], x1);
          F[r][1][2] = flux(h * (a1.z - a0.z), na1.y - a1.y, v23.y + x01.x, a0.y - my[r], m45.y + x1, nb1.y - b1.y,
                            v23.x, l0.y - ml[r], x4);
        }
      }
      {  // z edge
        const float h = ((v45.x + v45.y) + (x01.y + d23.y)) + (dxy0 + dxy2);
        const float hd = h * (na0.z - a0.z);
        F[r][2][2] = hd + hd;
        F[r][2][0] = flux(h * (na0.x - a0.x), nb0.z - na0.z, v45.x + d23.y, a0.z - l0.z, x01.y + dxy2, nb1.z - na1.z,
                          v45.y, am1.z - lm.z, dxy0);
        F[r][2][1] = flux(h * (na0.y - a0.y), na1.z - na0.z, v45.y + x01.y, a0.z - am1.z, d23.y + dxy0, nb1.z - nb0.z,
                          v45.x, l0.z - lm.z, dxy2);
      }
      if (r + 1 < FR) {  // the next row's row - 1
        am1 = a0;
        lm = l0;
        d23 = v23;
        dxy0 = x01.x;
        dxy2 = q[r * CP - 6 + 2];
        y3 = qm[r * CP + 3];
        y5 = m45.y;
      }
      ml[r] = l0.y;
    }
#pragma unroll
    for (int r = 0; r < FR; ++r) {
      mx[r + 1] = Pa[r].x;
      my[r] = Pa[r].y;
    }
    mx[0] = mx_next;
    if (full) {
#pragma unroll
      for (int c = 0; c < 3; ++c) fy[((w + 1) * 3 + c) * 32 + lane] = F[FR - 1][1][c];
    }
    if (w == kLeftWarp) {  // x edges from column -1 into column 0: lane j <-> row j
      const int j = lane & (FY - 1);
      const float* p = xs + s0 * 3 * VT + (j + 1) * VW;
      const float* pn = xs + s1 * 3 * VT + (j + 1) * VW;
      const float* u = cf + c0 * CT + (j + 1) * CP;
      const float* um = cf + cm * CT + (j + 1) * CP;
      const float ax = p[0], amx = p[-VW];
      if (full) {
        const float px = p[1], p1x = p[VW + 1], nx = pn[1], n1x = pn[VW + 1];
        const float v0 = u[0], v1 = u[1], dy2 = u[-CP + 2], m4 = um[4], l3 = um[-CP + 3], l5 = um[-CP + 5];
        const float h = ((v0 + v1) + (dy2 + m4)) + (l3 + l5);
        const float hd = h * (px - ax);
        const float f1 = flux(h * (p[VT + 1] - p[VT]), p1x - px, v0 + m4, ax - amx, dy2 + l5, n1x - nx, v1, lx1 - lx0, l3);
        const float f2 = flux(h * (p[2 * VT + 1] - p[2 * VT]), nx - px, v1 + dy2, ax - lx1, m4 + l3, n1x - p1x, v0,
                              amx - lx0, l5);
        if (lane < FY) {
          fxl[lane] = hd + hd;
          fxl[FY + lane] = f1;
          fxl[2 * FY + lane] = f2;
        }
      }
      lx1 = ax;
      lx0 = amx;
    }

    // epilogue values that are not staged: the previous iterate, the index of a stored-Galerkin stencil
    float e1[FR][3];
    int sv[FR];
    if ((MODE == ST_CHEB_STEP || STEN) && full) {
#pragma unroll
      for (int r = 0; r < FR; ++r) {
        const unsigned vo = (unsigned)(gv + r * nv + k * plane);
        sv[r] = -1;
        if ((r ? ok1 : ok0) && zin) {
          if (STEN) sv[r] = __ldg(op.sidx + vo);
          if (MODE == ST_CHEB_STEP) {
#pragma unroll
            for (int c = 0; c < 3; ++c) e1[r][c] = (a.xprev + c * V)[vo];
          }
        }
      }
    }
    __syncthreads();  // y and left x fluxes visible
    const float* ep = es + (k & 1) * (3 * NF * FX * FY) + threadIdx.x;
    if (full) {
#pragma unroll
      for (int r = 0; r < FR; ++r) {
        const bool in = (r ? ok1 : ok0) && zin;
        const int vo = gv + r * nv + k * plane;
        float g[3] = {0.f, 0.f, 0.f};
        if (STEN && sv[r] >= 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) g[c] = __ldg(op.ye + 3 * sv[r] + c);
        }
        const float xo[3] = {Pa[r].x, Pa[r].y, Pa[r].z};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float fl = __shfl_up_sync(0xffffffffu, F[r][0][c], 1);
          if (lane == 0) fl = fxl[c * FY + FR * w + r];
          const float f0 = r ? F[0][1][c] : fy[(w * 3 + c) * 32 + lane];  // y flux entering the row
          const float sum = ((fl - F[r][0][c]) + (f0 - F[r][1][c])) + (fz[r][c] - F[r][2][c]);
          float o = 0.f;
          if (in) {
            float eb = 0.f, ed = 0.f;
            if (NF > 0) {
              eb = ep[r * FNT + c * FX * FY];
              if (NF > 1) ed = ep[r * FNT + (3 + c) * FX * FY];
            }
            const float y = STEN ? fmaf(op.h6, sum, g[c]) : op.h6 * sum;
            if (MODE == ST_APPLY) {
              o = y;
            } else {
              const float res = STEN ? eb - y : fmaf(-op.h6, sum, eb);  // b - A x
              if (MODE == ST_RESID) o = res;
              if (MODE == ST_CHEB_FIRST) o = fmaf(a.s0, ed * res, xo[c]);
              if (MODE == ST_CHEB_STEP)
                o = fmaf(a.s1, ed * res, fmaf(a.s0, xo[c] - e1[r][c], xo[c]));
              if (MODE == ST_CHEB_PRE) o = fmaf(a.s1, ed * res, fmaf(a.s0, xo[c], xo[c]));
            }
          }
          if (col <= n && row + r <= n) put(vo, c, o);
        }
      }
    }
    // Dirichlet entries: plane 0, column 0 and row 0
    if (k == 0 && col <= n) {
#pragma unroll
      for (int r = 0; r < FR; ++r)
        if (row + r <= n)
          for (int c = 0; c < 3; ++c) put(gv + r * nv, c, 0.f);
    }
    if (ze >= 0 && (full || k == 0))
      for (int c = 0; c < 3; ++c) put(ze + k * plane, c, 0.f);
#pragma unroll
    for (int r = 0; r < FR; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) fz[r][c] = F[r][2][c];
    s0 = s1;
    c0 = c1;
  };
  // unrolled by two: the plane registers alternate roles
  for (int k = za - 1; k < zb; k += 2) {
    layer(k, A[0], B[0], A[1], B[1]);
    if (k + 1 >= zb) break;
    layer(k + 1, A[1], B[1], A[0], B[0]);
  }
  cpa_wait0();  // no copy may be in flight when the tile ends
}

template <int MODE, bool STEN, bool WIDE>
__global__ void __launch_bounds__(FNT, 2)
    stencil_f32_kernel(const LevelOp<float> op, const StencilArgs<float> a, const int zch, const int gx) {
  grid_dep_entry();
  extern __shared__ __align__(16) float sm_f32[];
  f32_block<MODE, STEN, WIDE>(op, a, zch, blockIdx.x % gx, blockIdx.x / gx, blockIdx.y, sm_f32);
}

// Batched form: a CTA per tile of up to N tasks, which come as kernel parameters:
// their fields are then read from the constant bank where they are used, as the
// single launch's.  Read from a device table or a copy in shared memory they
// stayed in registers across the march and spilled: the later step of twelve
// problems of 80^3 to 128^3 cubes took 597 us, 2.0 times the single launch's time
// per vertex.
template <int N>
struct F32Tasks {
  StencilTask<float, float> t[N];
  int n;
};
template <int MODE, bool STEN, bool WIDE, int N>
__global__ void __launch_bounds__(FNT, 2) stencil_f32_batch_kernel(const __grid_constant__ F32Tasks<N> p) {
  grid_dep_entry();
  extern __shared__ __align__(16) float sm_f32[];
  int q = 0;
  while (q + 1 < p.n && p.t[q + 1].tile0 <= (int64_t)blockIdx.x) ++q;
  const StencilTask<float, float>& tk = p.t[q];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;  // converged problem
  const int local = (int)((int64_t)blockIdx.x - tk.tile0), per = tk.tg.gxw * tk.tg.gyw;
  const int bz = local / per, u = local % per;
  f32_block<MODE, STEN, WIDE>(tk.op, tk.a, tk.tg.zch, u % tk.tg.gxw, u / tk.tg.gxw, bz, sm_f32);
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes, bool (&done)[64]) {
  int dev = 0;
  KL(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev]) {
    KL(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    done[dev] = true;
  }
  return cudaSuccess;
}

template <int MODE, bool STEN, bool WIDE = false>
cudaError_t launch_one(const LevelOp<float>& op, const StencilArgs<float>& a, const TileGrid& tg, cudaStream_t s) {
  static bool done[64] = {};
  KL(set_smem(stencil_f32_kernel<MODE, STEN, WIDE>, f32_smem<MODE>(), done));
  return launch_k(stencil_f32_kernel<MODE, STEN, WIDE>, dim3((unsigned)tg.per_z(), (unsigned)tg.gz), dim3(FNT), f32_smem<MODE>(),
                  s, op, a, tg.zch, tg.gxw);
}
template <int MODE, bool STEN, bool WIDE, int N>
cudaError_t launch_some(const StencilTask<float, float>* tasks, int n, cudaStream_t s) {
  static bool done[64] = {};
  KL(set_smem(stencil_f32_batch_kernel<MODE, STEN, WIDE, N>, f32_smem<MODE>(), done));
  F32Tasks<N> p{};
  p.n = n;
  int64_t tiles = 0;
  for (int i = 0; i < n; ++i) {
    p.t[i] = tasks[i];
    p.t[i].tile0 = tiles;
    tiles += (int64_t)tasks[i].tg.per_z() * tasks[i].tg.gz;
  }
  return launch_k(stencil_f32_batch_kernel<MODE, STEN, WIDE, N>, dim3((unsigned)tiles), dim3(FNT), f32_smem<MODE>(), s, p);
}
template <int MODE, bool STEN, bool WIDE = false>
cudaError_t launch_many(const StencilTask<float, float>* tasks, int ntasks, cudaStream_t s) {
  constexpr int N = kF32BatchTasks, S = 24;
  static_assert(sizeof(F32Tasks<N>) <= 32764, "kernel parameter limit");
  if (ntasks <= S) return launch_some<MODE, STEN, WIDE, S>(tasks, ntasks, s);
  for (int i = 0; i < ntasks; i += N) KL(launch_some<MODE, STEN, WIDE, N>(tasks + i, std::min(N, ntasks - i), s));
  return cudaSuccess;
}

}  // namespace

// Tiles over the vertices 1 .. n of each axis (coordinate 0 is written by the
// first tile).  Default z-chunk: the one with the least modelled time, whole
// waves of `slots` resident blocks times the planes a block marches (its
// chunk, the halo plane below and about one plane of prologue).
TileGrid f32_tiles(int n, int zch_req, int slots) {
  TileGrid g;
  g.gxw = (n + FX - 1) / FX;
  g.gyw = (n + FY - 1) / FY;
  g.x0n = n + 1;
  const int per = g.per_z(), sl = slots > 0 ? slots : 2 * 152;
  int zch = zch_req;
  if (zch <= 0) {
    double best = 1e300;
    for (int gz = 1; gz <= n; ++gz) {
      const int z = (n + gz - 1) / gz;
      if ((n + z - 1) / z != gz) continue;
      const double cost = (double)(((int64_t)per * gz + sl - 1) / sl) * (z + 2.0);
      if (cost < best - 1e-9) {
        best = cost;
        zch = z;
      }
    }
  }
  zch = std::min(std::max(zch, 1), n);
  g.gz = (n + zch - 1) / zch;
  g.zch = zch;
  return g;
}

cudaError_t launch_stencil_f32(int mode, const LevelOp<float>& op, const StencilArgs<float>& a, cudaStream_t s,
                               int zch_req) {
  int dev = 0, sms = 152;
  KL(cudaGetDevice(&dev));
  KL(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (op.n % 2) return cudaErrorInvalidValue;  // cube rows would not be 16-byte aligned (such levels are coarsest ones)
  const TileGrid tg = f32_tiles(op.n, zch_req, 2 * sms);
  const bool sten = op.sten != nullptr;
  if (a.out64 && mode != ST_CHEB_STEP) return cudaErrorInvalidValue;
  switch (mode) {
    case ST_APPLY: return sten ? launch_one<ST_APPLY, true>(op, a, tg, s) : launch_one<ST_APPLY, false>(op, a, tg, s);
    case ST_RESID: return sten ? launch_one<ST_RESID, true>(op, a, tg, s) : launch_one<ST_RESID, false>(op, a, tg, s);
    case ST_CHEB_FIRST:
      return sten ? launch_one<ST_CHEB_FIRST, true>(op, a, tg, s) : launch_one<ST_CHEB_FIRST, false>(op, a, tg, s);
    case ST_CHEB_STEP:  // ends the mixed cycle on the finest level, which has no stencils
      if (a.out64) return sten ? cudaErrorInvalidValue : launch_one<ST_CHEB_STEP, false, true>(op, a, tg, s);
      return sten ? launch_one<ST_CHEB_STEP, true>(op, a, tg, s) : launch_one<ST_CHEB_STEP, false>(op, a, tg, s);
    case ST_CHEB_PRE:
      return sten ? launch_one<ST_CHEB_PRE, true>(op, a, tg, s) : launch_one<ST_CHEB_PRE, false>(op, a, tg, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_stencil_f32_batch(int mode, bool sten, bool wide, const StencilTask<float, float>* tasks, int ntasks,
                                     cudaStream_t s) {
  if (ntasks <= 0) return cudaSuccess;
  if (wide && mode != ST_CHEB_STEP) return cudaErrorInvalidValue;
  switch (mode) {
    case ST_RESID:
      return sten ? launch_many<ST_RESID, true>(tasks, ntasks, s) : launch_many<ST_RESID, false>(tasks, ntasks, s);
    case ST_CHEB_FIRST:
      return sten ? launch_many<ST_CHEB_FIRST, true>(tasks, ntasks, s)
                  : launch_many<ST_CHEB_FIRST, false>(tasks, ntasks, s);
    case ST_CHEB_STEP:
      if (wide) return sten ? cudaErrorInvalidValue : launch_many<ST_CHEB_STEP, false, true>(tasks, ntasks, s);
      return sten ? launch_many<ST_CHEB_STEP, true>(tasks, ntasks, s)
                  : launch_many<ST_CHEB_STEP, false>(tasks, ntasks, s);
    case ST_CHEB_PRE:
      return sten ? launch_many<ST_CHEB_PRE, true>(tasks, ntasks, s) : launch_many<ST_CHEB_PRE, false>(tasks, ntasks, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace agca
