// window_f32_tc: the softmax window of the fp32 operator (Eq. 5, 6, 8) on the tensor cores, at fp32 precision.
//
// Every fp32 operand is split into three bf16 numbers, x = h + m + l (each rounded to nearest, so that l takes what 24
// bits leave), and a product is the six terms down to 2^-24: h h, h m, m h, m m, h l, l h.  bf16 products are exact in the
// fp32 accumulators; what is dropped is below 2^-26 of a product.  The accumulators round towards zero once per MMA, so
// the small terms go first and no sum runs longer than one key tile in TMEM: O of a tile is added to fp32 registers.
// The exponentials, maxima and row sums are those of window_simt.
// Relative error against 64 bits, 12 heads x 12,600 tokens of 128 channels: 3.0e-7, with window_simt 7.8e-7; ten other
// geometries 1.9 - 2.9e-7 against 1.9 - 4.0e-7.
//
//   Persistent: CTAs walk items (batch*head, chunk, tile of 128 queries), key tiles of 64.
//     warps 0-7   two threads per row (TMEM lane), each with 32 of a tile's keys and half of the output columns: Q into
//                 TMEM, softmax, split of P, sum of O, epilogue
//     warps 8-11  loaders: K and V rows from global memory, split, into swizzled shared-memory tiles (two stages)
//     warp 12     UMMA issuer: S = Q K^T (48 MMAs of N = 64), O = P V (24 of N = D), Q and P read from TMEM
//   TMEM: Q planes [0, 3D/2), two S slots of 96 columns (64 of S; the three planes of P overwrite them), O [3D/2 + 192, + D).
//   Q K^T of tile j + 1 is in the queue before P V of tile j, so that softmax j + 1 and the sum of O run beside MMAs.
// Bound by the MMAs: 3,072 cycles per key tile of 128 x 64 at D = 128.  The same layer: 4,783 -> 1,051 us (0.56 ms of MMAs).
//
// Values beyond 2^40 (or not finite) cannot be split safely: whoever sees one leaves the launch's epoch in *unsafe, and
// window_simt, launched behind this kernel, computes the call again; otherwise it ends at once.
#pragma once

#include "rehyat_simt.cuh"
#include "rehyat_tc_single.cuh"

namespace rehyat {

constexpr int F32_BN = 64, F32_STAGES = 2, F32_SOFTMAX_WARPS = 8, F32_LOAD_WARPS = 4;
constexpr int F32_THREADS = (F32_SOFTMAX_WARPS + F32_LOAD_WARPS + 1) * 32;
constexpr uint32_t F32_UNSAFE_BITS = 0x53800000u;     // 2^40

struct F32Bars {
  uint64_t q_ready, k_full[F32_STAGES], k_empty[F32_STAGES], v_full[F32_STAGES], v_empty[F32_STAGES];
  uint64_t s_ready[2], p_ready[2], pv_done, o_free, drained;
  uint32_t tmem_base;
  ptx::WaitCtx wctx;
  float mx[2][2][TC_BM];       // [key tile parity][half]: row maxima of the half's keys
  float ls[2][TC_BM];          // [half]: row sums
};
template <int D>
struct F32Shape {
  static constexpr int PLANE = F32_BN * D * 2, SUB = F32_BN * 128, STAGE = 6 * PLANE;    // K planes, then V planes
  static constexpr int SMEM = F32_STAGES * STAGE + (int)sizeof(F32Bars) + 16 + 1024;
  static constexpr uint32_t T_S = 3 * D / 2, T_O = T_S + 2 * 96;
};

// Two floats into the bf16 pairs of their three parts.
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = ptx::pack_bf16(x0, x1);
  x0 -= __uint_as_float(h << 16); x1 -= __uint_as_float(h & 0xffff0000u);
  m = ptx::pack_bf16(x0, x1);
  x0 -= __uint_as_float(m << 16); x1 -= __uint_as_float(m & 0xffff0000u);
  l = ptx::pack_bf16(x0, x1);
}
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t max_bits(uint32_t m, float4 x) {
  return max(max(m, max(abs_bits(x.x), abs_bits(x.y))), max(abs_bits(x.z), abs_bits(x.w)));
}

template <int D>
__global__ void __launch_bounds__(F32_THREADS, 1)
window_f32_tc(const float* q, const float* k, const float* v, float* out, Geo g, const float* rd, int rd_rows, float scale,
              int c_mode, ptx::WaitArgs wa, int n_items, int tiles, float* share, int wait_first, int* unsafe) {
  using namespace ptx;
  using SH = F32Shape<D>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t sb = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (sb - smem_u32(smem_raw));
  F32Bars* bars = reinterpret_cast<F32Bars*>(smem + F32_STAGES * SH::STAGE);
  const uint32_t wc = smem_u32(&bars->wctx);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bars->q_ready), F32_SOFTMAX_WARPS);
    for (int s = 0; s < F32_STAGES; ++s) {
      mbar_init(smem_u32(&bars->k_full[s]), F32_LOAD_WARPS); mbar_init(smem_u32(&bars->k_empty[s]), 1);
      mbar_init(smem_u32(&bars->v_full[s]), F32_LOAD_WARPS); mbar_init(smem_u32(&bars->v_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&bars->s_ready[s]), 1); mbar_init(smem_u32(&bars->p_ready[s]), F32_SOFTMAX_WARPS); }
    mbar_init(smem_u32(&bars->pv_done), 1); mbar_init(smem_u32(&bars->o_free), F32_SOFTMAX_WARPS);
    mbar_init(smem_u32(&bars->drained), 1);
    wait_ctx_init(&bars->wctx, wa);
    fence_mbar_init();
  }
  if (warp == 12) {
    tmem_alloc(smem_u32(&bars->tmem_base), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  if (wait_first) {                                                  // q, k, v may come from the direct predecessor
    grid_dep_wait();
    grid_dep_launch();
  }
  const auto n_tiles_of = [](const WinItem& w) { return (w.hi - w.lo + F32_BN - 1) / F32_BN; };

  if (warp >= 8 && warp < 12) {
    // ------------------------------------------------------------------ loaders
    constexpr int CH = D / 8, U = F32_BN * CH / 128;                 // 8-column chunks of a row; chunks per thread and tile
    const int t = threadIdx.x - 256;
    uint32_t n = 0, big = 0;                                         // key tiles so far; largest magnitude seen
    bool alive = !wa.withhold_loads;
    for (int item = blockIdx.x; item < n_items && alive; item += gridDim.x) {
      WinItem w;
      if (!win_item1(g, item, tiles, w)) continue;
      const long long hoff = head_offset(g, w.bh);
      const int n_kv = n_tiles_of(w);
      for (int j = 0; j < n_kv && alive; ++j, ++n) {
        const uint32_t st = n & 1, ph = (n >> 1) & 1;
#pragma unroll 1
        for (int kv = 0; kv < 2; ++kv) {
          const float* src = (kv ? v : k) + hoff;
          float4 x[U][2];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = t + 128 * u, key = w.lo + j * F32_BN + c / CH;
            const float* p = src + (long long)key * g.stride_n + (c % CH) * 8;
            x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (key < w.hi) { x[u][0] = ld4(p); x[u][1] = ld4(p + 4); }
          }
          alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(kv ? &bars->v_empty[st] : &bars->k_empty[st]), ph ^ 1, wc, TC_ERR_LOAD));
          if (!alive) break;
          const uint32_t dst = sb + st * SH::STAGE + kv * 3 * SH::PLANE;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = t + 128 * u;
            big = max_bits(max_bits(big, x[u][0]), x[u][1]);
            uint4 h, m, l;
            split3(x[u][0].x, x[u][0].y, h.x, m.x, l.x); split3(x[u][0].z, x[u][0].w, h.y, m.y, l.y);
            split3(x[u][1].x, x[u][1].y, h.z, m.z, l.z); split3(x[u][1].z, x[u][1].w, h.w, m.w, l.w);
            st_tile_chunk_sw128(dst, SH::SUB, c / CH, (c % CH) * 8, h);
            st_tile_chunk_sw128(dst + SH::PLANE, SH::SUB, c / CH, (c % CH) * 8, m);
            st_tile_chunk_sw128(dst + 2 * SH::PLANE, SH::SUB, c / CH, (c % CH) * 8, l);
          }
          fence_proxy_async_smem();
          mbar_arrive_warp(smem_u32(kv ? &bars->v_full[st] : &bars->k_full[st]), lane);
        }
      }
    }
    if (big >= F32_UNSAFE_BITS) *unsafe = wa.epoch;
  } else if (warp == 12) {
    // ------------------------------------------------------------------ UMMA issuer
    if (elect_one()) {
      constexpr uint32_t id_qk = idesc_bf16(TC_BM, F32_BN, 0, 0), id_pv = idesc_bf16(TC_BM, D, 0, 1);
      constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};   // planes of A and B, small terms first
      const uint64_t d_k = smem_desc_sw128(sb, 16, 1024), d_v = smem_desc_sw128(sb + 3 * SH::PLANE, SH::SUB, 1024);
      uint32_t n0 = 0, n_q = 0;                                      // key tiles of finished items, items
      bool alive = true;
      auto wait = [&](uint64_t* bar, uint32_t parity) {
        alive = alive && mbar_wait(smem_u32(bar), parity, wc, TC_ERR_MMA, TC_HINT_I);
        return alive;
      };
      for (int item = blockIdx.x; item < n_items && alive; item += gridDim.x) {
        WinItem w;
        if (!win_item1(g, item, tiles, w)) continue;
        const int n_kv = n_tiles_of(w);
        if (!wait(&bars->q_ready, n_q & 1)) break;
        ++n_q;
        auto qk = [&](uint32_t n) {                                  // key tile n (over all items) into slot n & 1
          const uint32_t st = n & 1;
          if (!wait(&bars->k_full[st], (n >> 1) & 1)) return;
          tc_fence_after();
          const uint64_t db = smem_desc_advance(d_k, st * SH::STAGE);
          const uint32_t acc = tmem + SH::T_S + st * 96;
#pragma unroll
          for (int t = 0; t < 6; ++t)
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              umma_ts(acc, tmem + PA[t] * (D / 2) + kk * 8, smem_desc_advance(db, PB[t] * SH::PLANE + (kk >> 2) * SH::SUB + (kk & 3) * 32),
                      id_qk, (t | kk) != 0);
          umma_commit(smem_u32(&bars->s_ready[st]));
          umma_commit(smem_u32(&bars->k_empty[st]));
        };
        qk(n0);
        if (n_kv > 1 && alive) qk(n0 + 1);
        for (int j = 0; j < n_kv && alive; ++j) {
          const uint32_t n = n0 + j, st = n & 1;
          if (!wait(&bars->v_full[st], (n >> 1) & 1) || !wait(&bars->p_ready[st], (n >> 1) & 1)) break;
          if (n > 0 && !wait(&bars->o_free, (n - 1) & 1)) break;     // O of the tile before has been read
          tc_fence_after();
          const uint64_t db = smem_desc_advance(d_v, st * SH::STAGE);
          const uint32_t pa = tmem + SH::T_S + st * 96;
#pragma unroll
          for (int t = 0; t < 6; ++t)
#pragma unroll
            for (int kk = 0; kk < F32_BN / 16; ++kk)
              umma_ts(tmem + SH::T_O, pa + PA[t] * (F32_BN / 2) + kk * 8, smem_desc_advance(db, PB[t] * SH::PLANE + kk * 2048), id_pv,
                      (t | kk) != 0);
          umma_commit(smem_u32(&bars->pv_done));
          umma_commit(smem_u32(&bars->v_empty[st]));
          if (j + 2 < n_kv) qk(n + 2);                               // into the slot this P V reads
        }
        n0 += n_kv;
      }
      // TMEM is not freed, nor does the CTA exit, with an MMA still running: this wait is not cut short by the abort flag
      umma_commit(smem_u32(&bars->drained));
      mbar_wait_drain(smem_u32(&bars->drained), 0, wc);
    }
  } else {
    // ------------------------------------------------------------------ softmax, sum of O, epilogue
    const int half = warp >> 2, r = (warp & 3) * 32 + lane;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16, tb = tmem + lane_off;
    // Waits that were given up return at once; these warps then run through the rest of their item (the barrier below
    // wants all eight) and leave together at the next item's head.  Nothing of an abandoned item is stored.
    auto wait = [&](uint64_t* bar, uint32_t parity) { mbar_wait(smem_u32(bar), parity, wc, TC_ERR_SOFTMAX); __syncwarp(); };
    auto barrier = [&](bool flag) -> bool {                          // of the eight warps; true if any thread's flag is
      uint32_t any;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                   : "=r"(any) : "r"((uint32_t)flag) : "memory");
      return any != 0;
    };
    uint32_t n = 0, big = 0;                                         // key tiles so far; largest magnitude of q
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
      WinItem w;
      if (!win_item1(g, item, tiles, w)) continue;
      if (barrier(wait_ctx_aborted(wc) != 0)) break;
      const int row = w.row_base + r, n_kv = n_tiles_of(w);
      const bool valid = row < w.q1;
      {
        // this thread's half of the row of Q into the three planes (every MMA that read the last ones is complete)
        const float* qp = q + q_row_offset(g, w.bh, valid ? row : w.row_base) + half * (D / 2);
#pragma unroll 1
        for (int c = 0; c < D / 2; c += 16) {
          uint32_t h[8], m[8], l[8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 x = valid ? ld4(qp + c + u * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
            big = max_bits(big, x);
            split3(x.x, x.y, h[2 * u], m[2 * u], l[2 * u]);
            split3(x.z, x.w, h[2 * u + 1], m[2 * u + 1], l[2 * u + 1]);
          }
          const uint32_t col = (half * (D / 2) + c) / 2;
          tmem_st8(tb + col, h); tmem_st8(tb + D / 2 + col, m); tmem_st8(tb + D + col, l);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive_warp(smem_u32(&bars->q_ready), lane);
      }
      float m = -INFINITY, l = 0.f, a_prev = 0.f;
      uint64_t o[D / 4];                                             // this thread's D/2 columns
#pragma unroll
      for (int c = 0; c < D / 4; ++c) o[c] = 0ull;
      auto add_o = [&](uint32_t nt, float alpha) {                   // o = o * alpha + O of key tile nt
        wait(&bars->pv_done, nt & 1);
        tc_fence_after();
        const uint64_t a2 = pk2(alpha, alpha);
#pragma unroll
        for (int c = 0; c < D / 2; c += 32) {
          uint32_t x[32];
          tmem_ld32(tb + SH::T_O + half * (D / 2) + c, x);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; e += 2) o[(c + e) / 2] = fma2(o[(c + e) / 2], a2, pk2u(x[e], x[e + 1]));
        }
        tc_fence_before();
        mbar_arrive_warp(smem_u32(&bars->o_free), lane);
      };
#pragma unroll 1
      for (int j = 0; j < n_kv; ++j, ++n) {
        const uint32_t st = n & 1;
        wait(&bars->s_ready[st], (n >> 1) & 1);
        tc_fence_after();
        uint32_t x[32];
        tmem_ld32(tb + SH::T_S + st * 96 + half * 32, x);
        tmem_wait_ld();
        const int n_here = w.hi - (w.lo + j * F32_BN + half * 32);   // keys of the window among this thread's
        float s[32], tmax = -INFINITY;
#pragma unroll
        for (int e = 0; e < 32; ++e) s[e] = __uint_as_float(x[e]) * scale;
        if (n_here < 32) {
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (e >= n_here) s[e] = -INFINITY;
        }
#pragma unroll
        for (int e = 0; e < 32; ++e) tmax = fmaxf(tmax, s[e]);
        bars->mx[st][half][r] = tmax;
        tc_fence_before();
        barrier(false);                                              // both halves have read S: P may overwrite it
        tc_fence_after();
        const float m_new = fmaxf(m, fmaxf(tmax, bars->mx[st][half ^ 1][r]));   // finite: the tile has a valid key
        const float alpha = expf(m - m_new);                         // exp(-inf) = 0 on the first tile
        m = m_new;
        float psum = 0.f;
        const uint32_t tp = tb + SH::T_S + st * 96 + half * 16;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t ph[8], pm[8], pl[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float p0 = expf(s[c * 16 + 2 * e] - m_new), p1 = expf(s[c * 16 + 2 * e + 1] - m_new);
            psum += p0 + p1;
            split3(p0, p1, ph[e], pm[e], pl[e]);
          }
          tmem_st8(tp + c * 8, ph); tmem_st8(tp + 32 + c * 8, pm); tmem_st8(tp + 64 + c * 8, pl);
        }
        l = l * alpha + psum;
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive_warp(smem_u32(&bars->p_ready[st]), lane);
        if (j > 0) add_o(n - 1, a_prev);
        a_prev = alpha;
      }
      add_o(n - 1, a_prev);
      bars->ls[half][r] = l;
      grid_dep_wait();                                               // the read-out is the predecessor's result
      grid_dep_launch();
      if (barrier(wait_ctx_aborted(wc) != 0)) break;
      l += bars->ls[half ^ 1][r];
      if (valid) {
        // Eq. 5, as in window_simt
        float ws = 1.f, lam = 0.f, nL = 0.f;
        if (w.linear) {
          lam = 1.f;
          if (c_mode == C_ZERO) {
            const float rr = fmaxf(m, 0.f);
            ws = expf(m - rr);
            lam = expf(-rr);
          }
          nL = rd[rd_index(g, rd_rows, D, w.bh, w.ci, row - w.q0, D / 4)];
        }
        const float inv = 1.f / (l * ws + lam * nL);
        if (share != nullptr && half == 0) share[(size_t)w.bh * g.N + row] = lam * nL * inv;
        float* orow = out + out_row_offset(g, w.bh, row) + half * (D / 2);
#pragma unroll
        for (int c = 0; c < D / 2; c += 4) {
          float4 aL = make_float4(0.f, 0.f, 0.f, 0.f);
          if (w.linear) aL = *reinterpret_cast<const float4*>(rd + rd_index(g, rd_rows, D, w.bh, w.ci, row - w.q0, (half * (D / 2) + c) >> 2));
          float y[4];
          upk2(o[c / 2], y[0], y[1]);
          upk2(o[c / 2 + 1], y[2], y[3]);
          st4(orow + c, (y[0] * ws + lam * aL.x) * inv, (y[1] * ws + lam * aL.y) * inv, (y[2] * ws + lam * aL.z) * inv,
              (y[3] * ws + lam * aL.w) * inv);
        }
      }
    }
    if (big >= F32_UNSAFE_BITS) *unsafe = wa.epoch;
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 12) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace rehyat
