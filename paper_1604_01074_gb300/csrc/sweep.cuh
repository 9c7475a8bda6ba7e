// Two-launch iteration for networks whose [Bbar; L] is sparse (SCHED_SWEEP), included by
// kernels.cu.
//
// With a null-space basis L in reduced form (host_factor) a water network's [Bbar; L] has
// three or four entries per row, so its two applications cost some hundred multiplications
// a node instead of 2 (n_x + n_u) n_v, and they fit into the tree passes around them.  What
// is left of the backward step is delta_n = Lambda_n r_n, one matrix per node.
//   tree_sweep    one CTA per chain or top node: v = path sums of delta, [Bbar; L] v, x and u,
//                 prox and dual update, w of the next iteration, then along the chain s, g =
//                 [Bbar; L]' [s; psi] and r bottom-up.
//   lambda_apply  delta_n = Lambda_n r_n, one warp per chain node; eight warps per top node,
//                 which first add up its r.  With S_m = xi_m + the s of m's chains and R_m =
//                 beta_m + the r of m's chains (m a top node),
//                   r_t = sum over the top nodes m below t, and t itself, of
//                         R_m + L' psi_m + c Bbar' S_m,
//                 c the number of top nodes from t down to m.  The last of m's chains and m
//                 itself forms the two terms in tree_sweep, so no top node waits for another.
// A general A: x and s along a chain take one product with A per node (A in shared memory, a
// block barrier each), and s and r of the top nodes climb in tree_sweep.  1531 nodes of a
// 50-tank network: 46 us an iteration, against 137 us of the six launches of schedule 2.
// Per iteration on GB300, one pack per node (the fastest of schedules 1 to 4): 2081 nodes 28 us in
// float32 (105), 117 us in float64 (388); 21 111 nodes 147 us (580), between events the tree pass
// 76 and Lambda 85; one pack for all of 21 111 nodes 107 us (401).  The tree pass is bound by issue
// slots (2 530 warp instructions a node, half of them the prox in float32 pairs), Lambda by HBM
// (439 MB, 5.9 TB/s without the gap before it) and in float64 by the pipe (2 lanes a cycle and SM).
// Vectors between the launches: h holds delta (n x n_v), rpub r of the chain nodes, spub s of
// the chain heads; a top node m's row of rpub holds R_m + L' psi_m, the first n_v entries of
// its row of wbuf (w, until the last arrival) Bbar' S_m.

// ---------------------------------------------------------------- sparse [Bbar; L]
// One entry: 8 bytes (float32) or 16 (float64).  Rows of K = [Bbar; L] and of K' are sorted
// by their entry count, so that the 32 rows a warp takes are of about one length.
template <typename VT>
struct SpEnt;
template <>
struct SpEnt<float> { float v; int c; };
template <>
struct SpEnt<double> { double v; long long c; };

template <typename VT>
__host__ __device__ inline int sp_bytes(int nnz, int n_k, int n_v) {
  return (int)round_up((long long)2 * nnz * sizeof(SpEnt<VT>) + (2ll * n_k + 2ll * n_v + 2) * sizeof(int), 16);
}
// put(r, e, (A x_r)_e + pre(r, e)) for rows r0 <= r < r1 of X (row stride xs) and all rows e
// of the sparse matrix.  A warp takes 32 rows e and four vectors r at a time, so each entry
// is read once for four products.  X has three readable rows behind r1.
template <int NW, typename VT, typename P, typename F>
__device__ __forceinline__ void sparse_rows(const SpEnt<VT>* ent, const int* ptr, const int* id, int rows, const VT* X,
                                            int xs, int r0, int r1, P&& pre, F&& put) {
  constexpr int NB = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rw = (rows + 31) / 32, ng = (r1 - r0 + NB - 1) / NB;
  for (int task = warp; task < rw * ng; task += NW) {
    const int g = task / rw, k = (task - g * rw) * 32 + lane;
    if (k >= rows) continue;
    const int e = id[k], rb = r0 + g * NB;
    VT acc[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] = rb + b < r1 ? pre(rb + b, e) : (VT)0;
    const VT* x = X + rb * xs;
    VT sum[NB] = {};
    const int q1 = ptr[k + 1];
    for (int q = ptr[k]; q < q1; ++q) {
      const SpEnt<VT> t = ent[q];
#pragma unroll
      for (int b = 0; b < NB; ++b) sum[b] += t.v * x[b * xs + (int)t.c];
    }
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (rb + b < r1) put(rb + b, e, sum[b] + acc[b]);
  }
}

__device__ __forceinline__ DS ld_state(const DS* p) {
  const float2 t = *reinterpret_cast<const float2*>(p);
  return {t.x, t.y};
}
__device__ __forceinline__ double ld_state(const double* p) { return *p; }
__device__ __forceinline__ void st_state(DS* p, DS v) { *reinterpret_cast<float2*>(p) = make_float2(v.hi, v.lo); }
__device__ __forceinline__ void st_state(double* p, double v) { *p = v; }

// acc += w v, the product taken exactly
__device__ __forceinline__ void st_fma_acc(DS& acc, float w, float v) { acc = st_axpy(acc, w, v); }
__device__ __forceinline__ void st_fma_acc(double& acc, double w, double v) { acc = fma(w, v, acc); }

// sums in the vector type or in the state type
template <typename ST, typename VT>
__device__ __forceinline__ ST to_sum(VT v) {
  if constexpr (std::is_same<ST, DS>::value)
    return DS{v, 0.f};
  else
    return v;
}
__device__ __forceinline__ void add_sum(DS& s, float v) {
  const DS t = two_sum(s.hi, v);
  s = fast_two_sum(t.hi, __fadd_rn(t.lo, s.lo));
}
__device__ __forceinline__ void add_sum(float& s, float v) { s += v; }
__device__ __forceinline__ void add_sum(double& s, double v) { s += v; }
__device__ __forceinline__ float sum_val(DS s) { return st_val(s); }
__device__ __forceinline__ float sum_val(float s) { return s; }
__device__ __forceinline__ double sum_val(double s) { return s; }

// Rows of the tree pass's vectors; in bfloat16 factors multiples of four entries, zero-padded,
// for the dense products below, whose [Bbar; L] has dense_kw words (two entries) a row: an odd
// number, so that 32 rows' words lie in 32 banks.
__host__ __device__ inline int sweep_pad(int n, bool b16) { return b16 ? (n + 3) / 4 * 4 : n; }
__host__ __device__ inline int dense_kw(int n_v) { return sweep_pad(n_v, true) / 2 | 1; }
template <typename VT>
__host__ __device__ inline size_t sweep_smem_bytes(int nnz, int depth, int n_x, int n_u, int n_v, bool general_A,
                                                   bool b16) {
  const int n_k = n_x + n_u, xk = sweep_pad(n_k, b16), xv = sweep_pad(n_v, b16);
  size_t b = sp_bytes<VT>(nnz, n_k, n_v);
  b += round_up((size_t)(3 * n_x + 2 * n_u) * sizeof(VT), 16);
  b += (size_t)(depth + 3) * (xv + xk) * sizeof(VT);  // depth + 3 >= 4 rows: the last arrival's too
  if (general_A) b += (size_t)n_x * n_x * sizeof(VT);
  if (b16) b += (size_t)xk * dense_kw(n_v) * sizeof(uint32_t);
  return round_up(b + (size_t)depth * sizeof(int), 16);
}

// Running maxima of absolute values as bit patterns, which order like the values; an
// infinity or NaN is above every finite one and stays visible in the maximum.  In float64 this
// also keeps comparisons and maxima off the float64 pipe (2 lanes a cycle and SM).
template <typename VT>
struct MaxAbs;
template <>
struct MaxAbs<float> {
  unsigned b = 0;
  __device__ void add(float v) { b = max(b, __float_as_uint(v) & 0x7fffffffu); }
  __device__ bool bad() const { return b >= 0x7f800000u; }
  __device__ float value() const { return __uint_as_float(b); }
};
template <>
struct MaxAbs<double> {
  unsigned long long b = 0;
  __device__ void add(double v) { b = max(b, (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull); }
  __device__ bool bad() const { return b >= 0x7ff0000000000000ull; }
  __device__ double value() const { return __longlong_as_double((long long)b); }
};

// st_val(st_sub(a, b)): the rounded sum of the difference's two terms is what renormalising them
// and adding them up again gives.
__device__ __forceinline__ float sub_val(DS a, DS b) {
  const DS t = two_sum(a.hi, -b.hi);
  return __fadd_rn(t.hi, __fadd_rn(t.lo, __fsub_rn(a.lo, b.lo)));
}
__device__ __forceinline__ double sub_val(double a, double b) { return a - b; }
// Signs of the tree pass: in float64 read from the bits, off the float64 pipe.
__device__ __forceinline__ bool sw_neg(DS x) { return x.hi < 0.f; }
__device__ __forceinline__ bool sw_neg(double x) { return __double_as_longlong(x) < 0; }
__device__ __forceinline__ bool sw_pos(DS x) { return x.hi > 0.f; }
__device__ __forceinline__ bool sw_pos(double x) { return __double_as_longlong(x) > 0; }
template <typename ST>
__device__ __forceinline__ ST sw_box(ST qh, ST ql) {
  return sw_pos(qh) ? qh : (sw_neg(ql) ? ql : st_from<ST>(0.0));
}

// Prox, dual update and w of node m (App. C; the arithmetic of Kern::warp_prox_staged) in two
// independent pieces, so that a node's work spreads over several warps: its tanks (both
// distance blocks, whose norms couple them) on one warp, 32 NT at most, and its inputs, 64 per
// warp.  z holds x and u on entry and w on return.  All loads are issued before the first use.
template <typename VT>
struct SweepOut {
  MaxAbs<VT> r, h, t;  // residual maxima: |x - t|, |x|, |t| of the prox
};
// Anchored solves (bfloat16 packs, B16): a delta launch takes w - w_a, exactly in the state
// type; an anchor stores w_a = w.
// All forms keep every operation of warp_prox_staged on the duals (the unnormalised float32
// extrapolation tried here had 1.4 times its mean error): in FORM 2 (the tensor-core path) the
// vectors are rounded to bfloat16 further on, where a last bit more or less turns into 2^-9.
template <typename VT, int NT, int FORM>
__device__ __forceinline__ void sweep_tanks(const IterArgs& a, int m, VT* z, const VT* bnd, int it, VT c, VT cn, int mode,
                                            SweepOut<VT>& o) {
  using ST = typename St<VT>::T;
  constexpr bool B16 = FORM != 0;
  const int lane = threadIdx.x & 31, n_x = a.n_x, nd = 2 * n_x + a.n_u;
  const VT *xs = bnd, *xhi = xs + n_x, *xlo = xhi + n_x;
  const ST* y1 = reinterpret_cast<const ST*>((it & 1) ? a.ybuf1 : a.ybuf0) + (long long)m * nd;
  ST* y2 = reinterpret_cast<ST*>((it & 1) ? a.ybuf0 : a.ybuf1) + (long long)m * nd;
  const ST zero = st_from<ST>(0.0);
  ST v1[NT], ws[NT], w1[NT], wz[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const int e = lane + 32 * k;
    v1[k] = ws[k] = w1[k] = wz[k] = zero;
    if (e < n_x) {
      v1[k] = ld_state(y1 + e);
      ws[k] = ld_state(y2 + e);
      w1[k] = ld_state(y1 + n_x + e);
      wz[k] = ld_state(y2 + n_x + e);
    }
  }
  VT wa[NT];
  if (B16)
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      const int e = lane + 32 * k;
      wa[k] = (mode & MODE_DELTA) && e < n_x ? reinterpret_cast<const VT*>(a.wa)[(long long)m * a.n_k + e] : (VT)0;
    }
  const VT ls = reinterpret_cast<const VT*>(a.step_s)[m], lz = reinterpret_cast<const VT*>(a.step_z)[m];
  const VT is = reinterpret_cast<const VT*>(a.inv_s)[m], iz = reinterpret_cast<const VT*>(a.inv_z)[m];
  const VT mus = reinterpret_cast<const VT*>(a.mu_s)[m], muz = (VT)a.gamma_d;
  VT* xo = reinterpret_cast<VT*>(a.xout) + (long long)m * n_x;
  // block norms ||lambda r|| of the two distance blocks
  VT ps = 0, pz = 0;
  ST qs[NT], qz[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const int e = lane + 32 * k;
    qs[k] = qz[k] = zero;
    if (e < n_x) {
      const VT x = z[e];
      ws[k] = st_extrap(v1[k], ws[k], c);
      wz[k] = st_extrap(w1[k], wz[k], c);
      const ST q = st_axpy(ws[k], ls, x - xs[e]);
      qs[k] = sw_neg(q) ? q : zero;  // C = {x >= x_s}
      qz[k] = sw_box(st_axpy(wz[k], lz, x - xhi[e]), st_axpy(wz[k], lz, x - xlo[e]));
      const VT rs = st_val(qs[k]), rz = st_val(qz[k]);
      ps += rs * rs;
      pz += rz * rz;
    }
  }
  // lanes 0 .. 15 add up and finish the s block, the others the z block: kappa = min(1, mu /
  // ||lambda r||), where a block within mu needs no root and division (in float64 as much work
  // as the rest of a node)
  const bool lo = lane < 16;
  VT sq = lo ? ps : pz;
  sq += __shfl_xor_sync(0xffffffffu, lo ? pz : ps, 16);
#pragma unroll
  for (int d = 8; d > 0; d >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, d);
  const VT mu = lo ? mus : muz;
  VT kap = 1;
  if (FORM == 2 || !(sq <= mu * mu)) {
    const VT dist = sqrt(sq);
    kap = dist > mu ? mu / dist : (VT)1;
  }
  const VT ks = __shfl_sync(0xffffffffu, kap, 0), kz = __shfl_sync(0xffffffffu, kap, 16);
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const int e = lane + 32 * k;
    if (e < n_x) {
      const VT x = z[e];
      const ST ysn = st_scale(qs[k], ks), yzn = st_scale(qz[k], kz);
      const VT es = sub_val(ysn, ws[k]) * is, ez = sub_val(yzn, wz[k]) * iz;
      st_state(y2 + e, ysn);
      st_state(y2 + n_x + e, yzn);
      xo[e] = x;
      if (B16 && (mode & MODE_DELTA)) {
        z[e] = st_val(st_sub(st_add(st_extrap(ysn, v1[k], cn), st_extrap(yzn, w1[k], cn)), st_from<ST>((double)wa[k])));
      } else {
        z[e] = st_extrap_val(ysn, v1[k], cn) + st_extrap_val(yzn, w1[k], cn);
        if (B16 && (mode & MODE_ANCHOR)) reinterpret_cast<VT*>(a.wa)[(long long)m * a.n_k + e] = z[e];
      }
      if (a.xbar) {  // ergodic average (theta_0 = 1: the previous contents are not read then)
        VT* b = reinterpret_cast<VT*>(a.xbar) + (long long)m * n_x + e;
        const VT th = (VT)a.theta[it];
        *b = it == 0 ? x : (VT)(((VT)1 - th) * *b + th * x);
      }
      o.r.add(es);  // a non-finite y shows in its residual
      o.r.add(ez);
      o.h.add(x);  // the prox maps a non-finite v to 0, so the primal iterate counts as well
      o.t.add(x - es);
      o.t.add(x - ez);
    }
  }
}
template <typename VT, int FORM>
__device__ __forceinline__ void sweep_inputs(const IterArgs& a, int m, int i0, VT* z, const VT* bnd, int it, VT c, VT cn,
                                             int mode, SweepOut<VT>& o) {
  using ST = typename St<VT>::T;
  constexpr bool B16 = FORM != 0;
  constexpr int NU = 2;
  const int lane = threadIdx.x & 31, n_x = a.n_x, n_u = a.n_u, nd = 2 * n_x + n_u;
  const VT *uhi = bnd + 3 * n_x, *ulo = uhi + n_u;
  const ST* y1 = reinterpret_cast<const ST*>((it & 1) ? a.ybuf1 : a.ybuf0) + (long long)m * nd + 2 * n_x;
  ST* y2 = reinterpret_cast<ST*>((it & 1) ? a.ybuf0 : a.ybuf1) + (long long)m * nd + 2 * n_x;
  const long long mu = (long long)m * n_u;
  const ST zero = st_from<ST>(0.0);
  ST p1[NU], p2[NU];
  VT lp[NU], ip[NU], wa[NU];
  const long long mk = (long long)m * a.n_k + n_x;
#pragma unroll
  for (int k = 0; k < NU; ++k) {
    const int i = i0 + lane + 32 * k;
    p1[k] = p2[k] = zero;
    lp[k] = ip[k] = 1;
    if (i < n_u) {
      p1[k] = ld_state(y1 + i);
      p2[k] = ld_state(y2 + i);
      lp[k] = reinterpret_cast<const VT*>(a.step_p)[mu + i];
      ip[k] = reinterpret_cast<const VT*>(a.inv_p)[mu + i];
      if (B16) wa[k] = (mode & MODE_DELTA) ? reinterpret_cast<const VT*>(a.wa)[mk + i] : (VT)0;
    }
  }
#pragma unroll
  for (int k = 0; k < NU; ++k) {
    const int i = i0 + lane + 32 * k;
    if (i < n_u) {
      const VT u = z[n_x + i];
      const ST wp = st_extrap(p1[k], p2[k], c);
      const ST ypn = sw_box(st_axpy(wp, lp[k], u - uhi[i]), st_axpy(wp, lp[k], u - ulo[i]));
      const VT ep = sub_val(ypn, wp) * ip[k];
      st_state(y2 + i, ypn);
      reinterpret_cast<VT*>(a.uout)[mu + i] = u;
      if (B16 && (mode & MODE_DELTA)) {
        z[n_x + i] = st_val(st_sub(st_extrap(ypn, p1[k], cn), st_from<ST>((double)wa[k])));
      } else {
        z[n_x + i] = st_extrap_val(ypn, p1[k], cn);
        if (B16 && (mode & MODE_ANCHOR)) reinterpret_cast<VT*>(a.wa)[mk + i] = z[n_x + i];
      }
      if (a.ubar) {
        VT* b = reinterpret_cast<VT*>(a.ubar) + mu + i;
        const VT th = (VT)a.theta[it];
        *b = it == 0 ? u : (VT)(((VT)1 - th) * *b + th * u);
      }
      o.r.add(ep);
      o.h.add(u);
      o.t.add(u - ep);
    }
  }
}

// In-place running sums of column `col` over rows r0, r0 + dr, ... (n of them); put(r, v) sees
// each sum.  Eight rows are read ahead of their sums.  The backward sums (s and r, ST the state
// type) run in two float32: their terms nearly cancel, and with them the error of x is a third
// of that with plain sums (1.0e-6 against 2.8e-6 after 60 iterations of 21 111 nodes).
template <typename ST, typename VT, typename F>
__device__ __forceinline__ void run_sums(VT* X, int xs, int col, int r0, int dr, int n, VT first, F&& put) {
  constexpr int B = 8;
  ST v = to_sum<ST>(first);
  for (int q0 = 0; q0 < n; q0 += B) {
    VT t[B];
#pragma unroll
    for (int b = 0; b < B; ++b) t[b] = q0 + b < n ? X[(r0 + (q0 + b) * dr) * xs + col] : (VT)0;
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (q0 + b < n) {
        add_sum(v, t[b]);
        put(r0 + (q0 + b) * dr, (VT)sum_val(v));
      }
  }
}

// Entries in pairs: two float32 in one register pair and one fused multiply-add instruction
// (f32x2), or one float64.
__device__ __forceinline__ unsigned long long f2(float x, float y) {
  return (unsigned long long)__float_as_uint(x) | ((unsigned long long)__float_as_uint(y) << 32);
}
struct PairF {
  using T = unsigned long long;
  static constexpr int N = 2;
  __device__ static T fma(T a, T b, T c) {
    T d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
  }
  __device__ static T dup(float x) { return f2(x, x); }
  __device__ static T zero() { return 0; }
  __device__ static float sum(T a) { return __uint_as_float((unsigned)a) + __uint_as_float((unsigned)(a >> 32)); }
  __device__ static float at(T a, int k) { return __uint_as_float((unsigned)(k ? a >> 32 : a)); }
  __device__ static void ld(const float* p, T (&o)[2]) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    o[0] = t.x;
    o[1] = t.y;
  }
};

// Two bfloat16 entries as a float32 pair
__device__ __forceinline__ unsigned long long bf2(uint32_t u) {
  return (unsigned long long)(u << 16) | ((unsigned long long)(u & 0xffff0000u) << 32);
}
// The dense [Bbar; L] of a bfloat16 factor (K: kw words a row) applied to float32 rows, four
// rows at a time.  Forward: put(r, e, (K V_r)_e), a lane per row e of K; the four rows' entries
// are broadcast reads, and pairs of products go through f32x2.  Backward: put(r, j, (K' Z_r)_j),
// two columns a lane.  They double the pass's instructions (about 550 and 800 a node at 177 x
// 97 entries), and still take less than streaming each node's own copy of K through the chains:
// 15 111 nodes of 18 stages 175 us an iteration, the pass 147 of them, against 433 with a chain
// pass of 366.
template <int NW, typename F>
__device__ __forceinline__ void dense_fwd(const uint32_t* K, int kw, int n_k, const float* V, int xv, int r0, int r1,
                                          F&& put) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ec = (n_k + 31) / 32, ng = (r1 - r0 + 3) / 4;
  for (int task = warp; task < ec * ng; task += NW) {
    const int g = task / ec, e = (task - g * ec) * 32 + lane, rb = r0 + 4 * g;
    const uint32_t* row = K + min(e, n_k - 1) * kw;
    unsigned long long acc[4] = {0, 0, 0, 0};
#pragma unroll 2
    for (int j = 0; j < xv; j += 4) {
      const unsigned long long k0 = bf2(row[j / 2]), k1 = bf2(row[j / 2 + 1]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(V + (rb + b) * xv + j);
        acc[b] = PairF::fma(k0, v.x, acc[b]);
        acc[b] = PairF::fma(k1, v.y, acc[b]);
      }
    }
    if (e < n_k)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (rb + b < r1) put(rb + b, e, PairF::sum(acc[b]));
  }
}
template <int NW, typename F>
__device__ __forceinline__ void dense_bwd(const uint32_t* K, int kw, int n_v, const float* Z, int xk, int r0, int r1,
                                          F&& put) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int jc = (n_v + 63) / 64, ng = (r1 - r0 + 3) / 4;
  for (int task = warp; task < jc * ng; task += NW) {
    const int g = task / jc, w = (task - g * jc) * 32 + lane, rb = r0 + 4 * g;
    const uint32_t* col = K + min(w, kw - 1);
    float acc[4][2] = {};
#pragma unroll 2
    for (int e = 0; e < xk; e += 4) {
      uint32_t u[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) u[i] = col[(e + i) * kw];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float4 y = *reinterpret_cast<const float4*>(Z + (rb + b) * xk + e);
        const float yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[b][0] += __uint_as_float(u[i] << 16) * yv[i];
          acc[b][1] += __uint_as_float(u[i] & 0xffff0000u) * yv[i];
        }
      }
    }
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (rb + b < r1 && 2 * w + h < n_v) put(rb + b, 2 * w + h, acc[b][h]);
  }
}

// out[e] += (A x)_e (trans: (A' x)_e) for e < n, A in shared memory: eight lanes a row.
template <int NW, typename VT>
__device__ __forceinline__ void add_Ax(const VT* A, int n, bool trans, const VT* x, VT* out) {
  const int lane = threadIdx.x & 31, part = lane & 7;
  for (int e0 = (threadIdx.x >> 5) * 4; e0 < n; e0 += NW * 4) {
    const int e = e0 + (lane >> 3);
    VT v = 0;
    if (e < n)
      for (int j = part; j < n; j += 8) v += (trans ? A[j * n + e] : A[e * n + j]) * x[j];
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if (part == 0 && e < n) out[e] += v;
  }
}

// NW warps a CTA at 64 registers a thread (float64: 128).  Most phases of a segment wait on
// memory or shared memory with few warps busy, so trees with several chains an SM run four
// small CTAs there, side by side in different phases; trees with at most a chain an SM have
// nothing to overlap and spread each chain over as many warps as an SM takes.
//
// FORM 0: float64 and float32 factors.  1: bfloat16 factors with a pack per node (see
// dense_fwd).  2: bfloat16 factors with one pack, whose products stay on the tensor cores:
// the first half of an iteration of schedule 2 in one launch - path sums of h, prox, s of every
// node - with the arithmetic of fwd_scan, prox_node and scan_kernel, in place of those three:
// 40 us instead of 73 on 13 830 nodes and 20 tanks, 72 instead of 108 on 15 876 nodes and 63.
template <typename VT>
__host__ __device__ inline size_t hsweep_smem_bytes(int depth, int n_x, int n_u) {
  const size_t b = round_up((size_t)(3 * n_x + 2 * n_u) * sizeof(VT), 16) + (size_t)3 * (depth + 3) * (n_x + n_u) * sizeof(VT);
  return round_up(b + (size_t)depth * sizeof(int), 16);
}
template <typename VT, int NT, int NW, int FORM>
__global__ void __launch_bounds__(32 * NW, NT == 8 ? 1 : (sizeof(VT) == 4 ? 32 : 16) / NW)
    tree_sweep(const __grid_constant__ IterArgs a, int nu, int mode) {
  using ST = typename St<VT>::T;
  constexpr int kSweepThreads = 32 * NW;
  constexpr bool B16 = FORM == 1, H = FORM == 2;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int flag[2];
  __shared__ VT red[3 * NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_x = a.n_x, n_u = a.n_u, n_k = a.n_k, n_v = a.n_v, nnz = H ? 0 : a.sp_nnz;
  const bool prox = (mode & MODE_PROX) != 0 && nu >= 1;
  // bfloat16 factors: the forward part continues a delta launch, the backward part is one
  // (both in the orthonormal basis of the packs); else they are the anchors' float32 ones
  const bool fd = B16 && !(mode & MODE_AFTER_ANCHOR), bd = B16 && (mode & MODE_DELTA) != 0;
  const int xv = sweep_pad(n_v, B16), xk = sweep_pad(n_k, B16);
  // ---- read while the previous launch drains: constants of the factor and the tree, and the
  // solve's affine data, complete before its first launch (nu = 0), which starts without
  // programmatic overlap
  const int blob = H ? 0 : sp_bytes<VT>(nnz, n_k, n_v);
  const SpEnt<VT>* ek = reinterpret_cast<const SpEnt<VT>*>(smem_raw);
  const SpEnt<VT>* et = ek + nnz;
  const int* rptr = reinterpret_cast<const int*>(et + nnz);
  const int *rid = rptr + n_k + 1, *cptr = rid + n_k, *cid = cptr + n_v + 1;
  VT* bnd = reinterpret_cast<VT*>(smem_raw + blob);
  VT* V = reinterpret_cast<VT*>(smem_raw + blob + round_up((3 * n_x + 2 * n_u) * (int)sizeof(VT), 16));  // delta, then v, then beta, g and r: a row of n_v per node
  VT* Z = H ? V : V + (a.depth + 3) * xv;  // e and u_hat, then x and u, then w and s: a row of n_k per node
  VT* HA = Z + (a.depth + 3) * xk;   // FORM 2: h_a, then e and u_hat, a row of n_k per node each
  VT* HE = HA + (a.depth + 3) * xk;
  VT* As = Z + (a.depth + 3) * xk;  // a general state matrix
  uint32_t* Kd = reinterpret_cast<uint32_t*>(As + (a.A ? n_x * n_x : 0));  // B16: the dense [Bbar; L]
  const int kw = dense_kw(n_v);
  int* sid = H ? reinterpret_cast<int*>(HE + (a.depth + 3) * xk) : reinterpret_cast<int*>(Kd + (B16 ? xk * kw : 0));
  if (B16) {
    const int ld = row_stride<__nv_bfloat16>(n_v);  // even
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.kd);
    if ((fd && prox) || bd)
      for (int q = tid; q < xk * kw; q += kSweepThreads) {
        const int e = q / kw, w = q - e * kw;
        Kd[q] = e < n_k && 2 * w < ld ? src[e * (ld / 2) + w] : 0u;  // the pack's padding is zero
      }
    for (int r = tid; r < a.depth + 3; r += kSweepThreads) {  // padding columns
      for (int j = n_v; j < xv; ++j) V[r * xv + j] = 0;
      for (int e = n_k; e < xk; ++e) Z[r * xk + e] = 0;
    }
  }
  if (a.A)
    for (int q = tid; q < n_x * n_x; q += kSweepThreads) As[q] = reinterpret_cast<const VT*>(a.A)[q];
  // chains first (the long tasks), then the top nodes
  const int b = (int)blockIdx.x < a.n_chains ? a.n_top + blockIdx.x : blockIdx.x - a.n_chains;
  const int4 d0 = *reinterpret_cast<const int4*>(a.seg + (long long)kSegInts * b);
  const int4 d1 = *reinterpret_cast<const int4*>(a.seg + (long long)kSegInts * b + 4);
  const int pl = d0.z, len = d1.y, tree = d0.w;
  const int L = pl + len;                  // the path (root .. parent), then the segment's own nodes
  const int own = len == 0 ? pl - 1 : pl;  // first own row (a top node ends its path)
  for (int r = tid; r < L; r += kSweepThreads) sid[r] = r < pl ? a.path_node[d0.y + r] : a.chain_node[d1.x + r - pl];
  for (int q = tid; q < blob / 16; q += kSweepThreads)
    reinterpret_cast<uint4*>(smem_raw)[q] = reinterpret_cast<const uint4*>(a.sp)[q];
  for (int q = tid; q < 3 * n_x + 2 * n_u; q += kSweepThreads) {
    const void* src = q < n_x ? a.x_s : q < 2 * n_x ? a.x_max : q < 3 * n_x ? a.x_min : q < 3 * n_x + n_u ? a.u_max : a.u_min;
    const int i = q < 3 * n_x ? q % n_x : (q - 3 * n_x) % n_u;
    bnd[q] = reinterpret_cast<const VT*>(src)[i];
  }
  const VT c = (VT)a.cvec[prox ? nu - 1 : nu], cn = prox ? (VT)a.cvec[nu] : (VT)0;
  __syncthreads();
  if (prox && !fd) {
    const VT* E = reinterpret_cast<const VT*>(a.e);
    const VT* UH = reinterpret_cast<const VT*>(a.uhat);
    for (int r = warp; r < L; r += NW) {
      const long long m = sid[r];
      VT* to = (H ? HE : Z) + r * xk;
      for (int e = lane; e < n_x; e += 32) cp_async_elem(to + e, E + m * n_x + e);
      if (r >= own)
        for (int i = lane; i < n_u; i += 32) cp_async_elem(to + n_x + i, UH + m * n_u + i);
    }
  }
  if (prox && fd)  // the anchor's x and u, read behind the path sums: towards the L2
    for (int r = own + warp; r < L; r += NW)
      for (int e = 32 * lane; e < n_k; e += 32 * 32) {
        const long long at = (long long)sid[r] * n_k + e;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const VT*>(a.ha) + at));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const VT*>(a.ha_lo) + at));
      }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (prox) {
    const VT* delta = reinterpret_cast<const VT*>(a.h);
    if (H)
      for (int r = warp; r < L; r += NW)
        for (int e = lane; e < n_k; e += 32) {
          cp_async_elem(Z + r * xk + e, delta + (long long)sid[r] * n_k + e);
          cp_async_elem(HA + r * xk + e, reinterpret_cast<const VT*>(a.ha) + (long long)sid[r] * n_k + e);
        }
    for (int r = H ? L : warp; r < L; r += NW)
      for (int j = lane; j < n_v; j += 32) cp_async_elem(V + r * xv + j, delta + (long long)sid[r] * n_v + j);
  }
  const bool stop = early_exit(a, nu, mode, flag, true) || !tree_active(a, tree, nu);
  cp_async_wait_all();
  // the solve stopped, or this tree of a forest did (it keeps its iterates)
  if (stop) return;
  SweepOut<VT> o;
  if (prox) {
    __syncthreads();
    if (H) {  // path sums of h + h_a, as in fwd_scan
      for (int e = tid; e < n_k; e += kSweepThreads) {
        VT v = 0, x = e < n_x ? reinterpret_cast<const VT*>(a.p0)[(long long)tree * n_x + e] : (VT)0;
#pragma unroll 4
        for (int r = 0; r < L; ++r) {
          v += Z[r * xk + e] + HA[r * xk + e];
          const VT ev = e < n_x || r >= own ? HE[r * xk + e] : (VT)0;
          if (e < n_x)
            x += v + ev;
          else
            x = v + ev;
          Z[r * xk + e] = x;
        }
      }
      __syncthreads();
    } else if (B16 && !fd) {
      // The base of the delta launches up to the next anchor, in two float32 throughout (ha,
      // ha_lo): rounded to one, the same error would enter the duals in each of them.
      if (tid < n_k) {
        const int e = rid[tid], q0 = rptr[tid], q1 = rptr[tid + 1];
        ST inc = st_from<ST>(0.0), x = to_sum<ST>(e < n_x ? reinterpret_cast<const VT*>(a.p0)[(long long)tree * n_x + e] : (VT)0);
        for (int r = 0; r < L; ++r) {
          for (int q = q0; q < q1; ++q) st_fma_acc(inc, ek[q].v, V[r * xv + (int)ek[q].c]);
          if (e >= n_x) x = to_sum<ST>((VT)0);  // u_n = L v_n + u_hat_n, x_n = x_parent + Bbar v_n + e_n
          if (e < n_x || r >= own) add_sum(x, Z[r * xk + e]);
          x = st_add(x, inc);
          Z[r * xk + e] = st_val(x);
          if (r >= own) {
            reinterpret_cast<VT*>(a.ha)[(long long)sid[r] * n_k + e] = st_val(x);
            reinterpret_cast<VT*>(a.ha_lo)[(long long)sid[r] * n_k + e] = st_val(st_sub(x, to_sum<ST>(st_val(x))));
          }
        }
      }
      __syncthreads();
    } else {
      if (tid < n_v)  // v along the path
        run_sums<VT>(V, xv, tid, 0, 1, L, (VT)0, [&](int r, VT v) { V[r * xv + tid] = v; });
      __syncthreads();
      // x increments (Bbar v + e) and u; of path nodes only the tanks are used
      if constexpr (B16)
        dense_fwd<NW>(Kd, kw, n_k, V, xv, 0, L, [&](int r, int e, VT v) { Z[r * xk + e] = v; });
      else
        sparse_rows<NW, VT>(
            ek, rptr, rid, n_k, V, xv, 0, L, [&](int r, int e) -> VT { return Z[r * xk + e]; },
            [&](int r, int e, VT v) { Z[r * xk + e] = v; });
      __syncthreads();
      if (a.A) {  // x_n = A x_parent + Bbar v_n + e_n (App. B), a barrier a node
        if (tid < n_x) Z[L * xk + tid] = reinterpret_cast<const VT*>(a.p0)[(long long)tree * n_x + tid];
        for (int r = 0; r < L; ++r) {
          __syncthreads();
          add_Ax<NW>(As, n_x, false, Z + (r > 0 ? r - 1 : L) * xk, Z + r * xk);
        }
      } else if (tid < n_x)  // x_n = x_parent + Bbar v_n + e_n
        run_sums<VT>(Z, xk, tid, 0, 1, L, B16 ? (VT)0 : reinterpret_cast<const VT*>(a.p0)[(long long)tree * n_x + tid],
                     [&](int r, VT v) { Z[r * xk + tid] = v; });
      __syncthreads();
      if (B16) {  // the linear part on the anchor's x and u
        for (int r = own + warp; r < L; r += NW)
          for (int e = lane; e < n_k; e += 32) {
            const long long at = (long long)sid[r] * n_k + e;
            ST x = to_sum<ST>(reinterpret_cast<const VT*>(a.ha)[at]);
            add_sum(x, reinterpret_cast<const VT*>(a.ha_lo)[at]);
            add_sum(x, Z[r * xk + e]);
            Z[r * xk + e] = sum_val(x);
          }
        __syncthreads();
      }
    }
  }
  if (!H && len > 0 && (mode & MODE_BWD) && !bd) {  // beta, used after the prox
    const VT* beta = reinterpret_cast<const VT*>(a.beta);
    for (int r = own + warp; r < L; r += NW)
      for (int j = lane; j < n_v; j += 32) cp_async_elem(V + r * xv + j, beta + (long long)sid[r] * n_v + j);
  }
  if (prox) {
    const int rows = L - own, ni = (n_u + 63) / 64;
    for (int task = warp; task < rows * (1 + ni); task += NW) {
      if (task < rows) {
        const int r = own + task;
        sweep_tanks<VT, NT, FORM>(a, sid[r], Z + r * xk, bnd, nu - 1, c, cn, mode, o);
      } else {
        const int q = (task - rows) / ni, r = own + q;
        sweep_inputs<VT, FORM>(a, sid[r], 64 * (task - rows - q * ni), Z + r * xk, bnd, nu - 1, c, cn, mode, o);
      }
    }
    if (o.r.bad() || o.h.bad()) a.flags[1] = SMPC_EDIVERGED;
  } else {  // w^nu without a prox: the first iteration
    const int nd = 2 * n_x + n_u;
    for (int r = own + warp; r < L; r += NW) {
      const ST* ya = reinterpret_cast<const ST*>((nu & 1) ? a.ybuf1 : a.ybuf0) + (long long)sid[r] * nd;
      const ST* yb = reinterpret_cast<const ST*>((nu & 1) ? a.ybuf0 : a.ybuf1) + (long long)sid[r] * nd;
      for (int e = lane; e < n_k; e += 32) {
        if (e < n_x)
          Z[r * xk + e] = st_val(st_add(st_extrap(ld_state(ya + e), ld_state(yb + e), c),
                                         st_extrap(ld_state(ya + n_x + e), ld_state(yb + n_x + e), c)));
        else
          Z[r * xk + e] = st_val(st_extrap(ld_state(ya + n_x + e), ld_state(yb + n_x + e), c));
        if (FORM != 0) reinterpret_cast<VT*>(a.wa)[(long long)sid[r] * n_k + e] = Z[r * xk + e];  // the first launch anchors
      }
    }
  }
  if (prox) {  // residual maxima (Sec. IV-E)
    const VT rw = warp_max(o.r.value()), hw = warp_max(o.h.value()), tw = warp_max(o.t.value());
    if (lane == 0) {
      red[warp] = rw;
      red[NW + warp] = hw;
      red[2 * NW + warp] = tw;
    }
  }
  cp_async_wait_all();
  __syncthreads();
  if (prox && tid >= kSweepThreads - 3) {
    const int k = kSweepThreads - 1 - tid;
    VT v = 0;
    for (int w = 0; w < NW; ++w) v = fmax(v, red[k * NW + w]);
    atomic_max_nonneg(a.res + 3ll * (nu - 1) + k, (double)v);
    if (a.res_tree) atomic_max_nonneg(a.res_tree + 3ll * ((long long)(nu - 1) * a.R + tree) + k, (double)v);
  }
  if (!(mode & MODE_BWD)) return;
  if constexpr (H) {  // w and s of every node (scan_kernel's sums); the top nodes' by last arrival
    VT* S = reinterpret_cast<VT*>(a.spub);
    for (int r = own + warp; r < L; r += NW)
      for (int e = lane; e < n_k; e += 32) reinterpret_cast<VT*>(a.wbuf)[(long long)sid[r] * n_k + e] = Z[r * xk + e];
    if (len > 0 && tid < n_x)
      run_sums<VT>(Z, xk, tid, L - 1, -1, len, (VT)0, [&](int r, VT v) { S[(long long)sid[r] * n_x + tid] = v; });
    for (int t = d0.x; t >= 0; t = a.parent[t]) {
      __syncthreads();
      if (tid == 0) {
        fence_acq_rel_gpu();
        const int last = atomicAdd(&a.counters[t], 1) == a.top_expect[t] - 1;
        if (last) {
          a.counters[t] = 0;
          fence_acq_rel_gpu();
        }
        flag[1] = last;
      }
      __syncthreads();
      if (!flag[1]) return;
      const int c0 = a.child_begin[t], cc = a.child_count[t];
      for (int e = tid; e < n_x; e += kSweepThreads) {
        VT v = ldcg(reinterpret_cast<const VT*>(a.wbuf) + (long long)t * n_k + e);
        constexpr int C = 8;
        for (int i = 0; i < cc; i += C) {
          VT u[C];
#pragma unroll
          for (int k = 0; k < C; ++k) u[k] = i + k < cc ? ldcg(S + (long long)(c0 + i + k) * n_x + e) : (VT)0;
#pragma unroll
          for (int k = 0; k < C; ++k)
            if (i + k < cc) v += u[k];
        }
        S[(long long)t * n_x + e] = v;
      }
    }
    return;
  }
  if (len == 0) {  // a top node: its w
    VT* w = reinterpret_cast<VT*>(a.wbuf) + (long long)sid[own] * n_k;
    for (int e = tid; e < n_k; e += kSweepThreads) w[e] = Z[own * xk + e];
  } else {
    if (a.A) {  // s_n = xi_n + A' s_child
      for (int r = L - 2; r >= own; --r) {
        add_Ax<NW>(As, n_x, true, Z + (r + 1) * xk, Z + r * xk);
        __syncthreads();
      }
      if (tid < n_x) reinterpret_cast<VT*>(a.spub)[(long long)sid[own] * n_x + tid] = Z[own * xk + tid];
    } else if (tid < n_x) {  // s along the chain, bottom-up
      VT s = 0;
      run_sums<ST>(Z, xk, tid, L - 1, -1, len, (VT)0, [&](int r, VT v) { Z[r * xk + tid] = s = v; });
      reinterpret_cast<VT*>(a.spub)[(long long)sid[own] * n_x + tid] = s;
    }
    __syncthreads();
    if constexpr (B16) {
      if (bd) dense_bwd<NW>(Kd, kw, n_v, Z, xk, own, L, [&](int r, int j, VT v) { V[r * xv + j] = v; });
    }
    if (!bd) sparse_rows<NW, VT>(
        et, cptr, cid, n_v, Z, xk, own, L, [&](int r, int j) -> VT { return V[r * xv + j]; },
        [&](int r, int j, VT v) { V[r * xv + j] = v; });
    __syncthreads();
    if (tid < n_v) {  // r along the chain
      VT* R = reinterpret_cast<VT*>(a.rpub);
      run_sums<ST>(V, xv, tid, L - 1, -1, len, (VT)0, [&](int r, VT v) { R[(long long)sid[r] * n_v + tid] = v; });
    }
  }
  // The last of a top node and its chains forms the node's two terms of r.  With a general A
  // (s_t = xi_t + A' sum_c s_c) they are no plain sums: there the last of a top node and all
  // its children forms its s and r, and climbs on.
  const VT* sp = reinterpret_cast<const VT*>(a.spub);
  VT* rp = reinterpret_cast<VT*>(a.rpub);
  VT *Z0 = Z, *Z1 = Z + xk, *R0 = Z + 2 * xk;
  const bool climb = a.A != nullptr;
  for (int t = d0.x; t >= 0; t = climb ? a.parent[t] : -1) {
    __syncthreads();  // this CTA's outputs, then one fence, before its arrival
    if (tid == 0) {
      fence_acq_rel_gpu();
      const int last = atomicAdd(&a.counters[t], 1) == (climb ? a.top_expect[t] - 1 : a.chain_kids[t]);
      if (last) {
        a.counters[t] = 0;
        fence_acq_rel_gpu();
      }
      flag[1] = last;
    }
    __syncthreads();
    if (!flag[1]) return;
    const int c0 = a.child_begin[t], cc = a.child_count[t];
    VT* wt = reinterpret_cast<VT*>(a.wbuf) + (long long)t * n_k;
    // row 0: [S; 0] and row 1: [0; psi]; with A row 0: [xi; psi] and row 1 the children's s.
    // Row 2: beta and the children's r
    for (int e = n_x + tid; e < n_k; e += kSweepThreads) {
      Z1[e] = ldcg(wt + e);
      Z0[e] = climb ? Z1[e] : (VT)0;
    }
    for (int q = tid; q < n_x + n_v; q += kSweepThreads) {
      const bool tank = q < n_x;
      const VT* in = tank ? sp : rp;
      const int cols = tank ? n_x : n_v, e = tank ? q : q - n_x;
      const VT own_w = tank ? ldcg(wt + e) : reinterpret_cast<const VT*>(a.beta)[(long long)t * n_v + e];
      ST sum = st_from<ST>(0.0);
      if (!(climb && tank) && (tank || !bd)) st_fma_acc(sum, (VT)1, own_w);
      constexpr int C = 8;
      for (int i = 0; i < cc; i += C) {  // children in index order, C loads in flight
        VT v[C];
#pragma unroll
        for (int k = 0; k < C; ++k)
          v[k] = i + k < cc && (climb || a.top_expect[c0 + i + k] == 0) ? ldcg(in + (long long)(c0 + i + k) * cols + e)
                                                                        : (VT)0;
#pragma unroll
        for (int k = 0; k < C; ++k) st_fma_acc(sum, (VT)1, v[k]);
      }
      if (!tank) {
        R0[e] = st_val(sum);
      } else {
        Z0[e] = climb ? own_w : st_val(sum);
        Z1[e] = climb ? st_val(sum) : (VT)0;
      }
    }
    __syncthreads();  // also: w has been read
    if (climb) {
      add_Ax<NW>(As, n_x, true, Z1, Z0);
      __syncthreads();
      if (tid < n_x) reinterpret_cast<VT*>(a.spub)[(long long)t * n_x + tid] = Z0[tid];
    }
    if constexpr (B16) {
      if (bd)
        dense_bwd<NW>(Kd, kw, n_v, Z, xk, 0, 2, [&](int r, int j, VT v) {
          if (r == 1)
            rp[(long long)t * n_v + j] = v + R0[j];
          else
            wt[j] = v;
        });
    }
    if (!bd) sparse_rows<NW, VT>(
        et, cptr, cid, n_v, Z, xk, 0, climb ? 1 : 2, [&](int r, int j) -> VT { return climb || r == 1 ? R0[j] : (VT)0; },
        [&](int r, int j, VT v) { (climb || r == 1 ? rp + (long long)t * n_v : wt)[j] = v; });
  }
}

// ---------------------------------------------------------------- delta = Lambda r
// Lambda_n = Lambda / (2 p_n) is symmetric; each node keeps one half of it, as blocks of BS x
// BS entries (BS = 4, or 8 when n_v > 128) on "circulant diagonals": with G = n_v / BS block
// rows, diagonal k holds the blocks (I, (I + k) mod G) of all I, k = 0 .. G / 2 (for an even G
// the last diagonal holds the first G / 2 of them).  Lane I takes block (I, I + k) in step k
// and uses it twice: for row block I, kept in registers, and transposed for row block I + k,
// whose sums travel from lane to lane.  A step's blocks are stored chunk by chunk (16 bytes
// of every lane's block side by side), so that each load instruction of a warp reads one
// contiguous piece.  Half the bytes of the square layout: what bounds the launch on trees
// that do not fit the cache.
__host__ __device__ inline int lam_bs(int n_v) { return n_v <= 128 ? 4 : 8; }
__host__ __device__ inline long long lam_entries(int n_v) {
  const int bs = lam_bs(n_v), G = (n_v + bs - 1) / bs;
  return (long long)(G / 2 + 1) * G * bs * bs;
}

template <typename MT>
__global__ void lam_pack_kernel(int n, int n_v, const double* Lam, const double* prob, MT* out) {
  constexpr int CE = 16 / (int)sizeof(MT);
  const int bs = lam_bs(n_v), G = (n_v + bs - 1) / bs, nc = bs * bs / CE;
  const long long per = lam_entries(n_v);
  for (int m = blockIdx.x; m < n; m += gridDim.x) {
    const double inv = prob ? 1.0 / (2.0 * prob[m]) : 1.0;
    for (int q = threadIdx.x; q < per; q += blockDim.x) {
      const int t = q % CE, I = (q / CE) % G, c = (q / CE / G) % nc, k = q / CE / G / nc;
      const int at = c * CE + t, J = (I + k) % G;
      const int i = bs * I + at / bs, j = bs * J + at % bs;
      const bool half = 2 * k == G && I >= G / 2;  // the pair (I, I + G / 2) is kept once
      out[m * per + q] = (MT)(i < n_v && j < n_v && !half ? Lam[(long long)i * n_v + j] * inv : 0.0);
    }
  }
}

// Steps [k0, k1) of one matrix (in shared or global memory) on a warp: acc += the part of
// Lambda r in row block `lane`.  rs: r, zero-padded to G BS entries, 16-byte aligned.
struct PairD {
  using T = double;
  static constexpr int N = 1;
  __device__ static T fma(T a, T b, T c) { return ::fma(a, b, c); }
  __device__ static T dup(double x) { return x; }
  __device__ static T zero() { return 0; }
  __device__ static double sum(T a) { return a; }
  __device__ static double at(T a, int) { return a; }
  __device__ static void ld(const double* p, T (&o)[2]) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    o[0] = t.x;
    o[1] = t.y;
  }
};
template <typename VT, int BS, typename MT>
__device__ __forceinline__ void lam_steps(const MT* lam, int G, const VT* rs, int k0, int k1, VT (&out)[BS]) {
  using P = typename std::conditional<sizeof(VT) == 4, PairF, PairD>::type;
  using T = typename P::T;
  constexpr int CE = 16 / (int)sizeof(VT);  // entries of a chunk: two pairs
  constexpr int NC = BS * BS / CE, RC = BS / CE > 0 ? BS / CE : 1, NP = BS / P::N;
  const int lane = threadIdx.x & 31;
  const int I = lane < G ? lane : 0;  // idle lanes repeat lane 0's loads; nothing of theirs is used
  T ri[BS], acc[BS], tr[NP];
#pragma unroll
  for (int r = 0; r < BS; ++r) {
    ri[r] = P::dup(rs[BS * I + r]);
    acc[r] = P::zero();
  }
#pragma unroll
  for (int q = 0; q < NP; ++q) tr[q] = P::zero();
  const int from = I + 1 < G ? I + 1 : 0;
  // a 16-byte chunk of the matrix: CE entries, or two times CE in bfloat16
  constexpr int ME = 16 / (int)sizeof(MT), MC = BS * BS / ME;
  const MT* blk = lam + ((long long)k0 * MC * G + I) * ME;
  int J = I + k0 < G ? I + k0 : I + k0 - G;
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    T A[NC][2], rj[RC][2];
#pragma unroll
    for (int c = 0; c < MC; ++c) {
      if constexpr (sizeof(MT) == 2) {
        const uint4 u = *reinterpret_cast<const uint4*>(blk + (long long)c * G * ME);
        A[2 * c][0] = bf2(u.x);
        A[2 * c][1] = bf2(u.y);
        A[2 * c + 1][0] = bf2(u.z);
        A[2 * c + 1][1] = bf2(u.w);
      } else {
        P::ld(blk + (long long)c * G * ME, A[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < RC; ++c) P::ld(rs + BS * J + c * CE, rj[c]);
    blk += (long long)MC * G * ME;
    if (++J == G) J = 0;
    if (k > 0) {  // the diagonal blocks are symmetric themselves
#pragma unroll
      for (int q = 0; q < NP; ++q) tr[q] = __shfl_sync(0xffffffffu, tr[q], from);
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) tr[(c % RC) * 2 + h] = P::fma(A[c][h], ri[c / RC], tr[(c % RC) * 2 + h]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) acc[c / RC] = P::fma(A[c][h], rj[c % RC][h], acc[c / RC]);
  }
  int back = (I - (k1 - 1)) % G;  // row block I's travelling sums are on lane I - (k1 - 1)
  if (back < 0) back += G;
#pragma unroll
  for (int q = 0; q < NP; ++q) tr[q] = __shfl_sync(0xffffffffu, tr[q], back);
#pragma unroll
  for (int r = 0; r < BS; ++r) out[r] = P::sum(acc[r]) + P::at(tr[r / P::N], r % P::N);
}

constexpr int kTopList = 128;  // <= 256
__device__ __forceinline__ void bar_top() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// Warps 0 .. LW - 1 of a CTA take chain nodes, warps LW .. LW + 7 the top nodes, side by side.
// A chain warp owns one slot of shared memory, filled by a bulk copy of its next node's
// matrix: the first copy is issued before the previous launch has drained (the matrices are
// constants), the following ones as soon as the slot has been read, and with eight warps on an
// SM (two CTAs) seven copies are in flight while one is used.  One matrix shared by all nodes
// is copied once per CTA.  slots = 0: a matrix larger than shared memory is read in place.
template <typename VT, typename MT>
__host__ __device__ inline size_t lambda_smem_bytes(int n_v, int slots) {
  return (size_t)round_up((size_t)slots * lam_entries(n_v) * sizeof(MT), 128) + (size_t)kWarps * 32 * kStateSize +
         (size_t)kWarps * 32 * lam_bs(n_v) * sizeof(VT);
}

template <typename VT, typename MT, int BS, int LW>
__global__ void __launch_bounds__((LW + 8) * 32, BS == 4 && sizeof(VT) == 4 ? 2 : 1)
    lambda_apply(const __grid_constant__ IterArgs a, int slots, int nu, int mode) {
  using ST = typename St<VT>::T;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int flag[2];
  __shared__ __align__(16) VT rs[LW + 1][32 * BS];
  __shared__ uint64_t bar[LW];
  __shared__ int2 list[kTopList];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_x = a.n_x, n_k = a.n_k, n_v = a.n_v, n_c = a.A ? a.n : a.n - a.n_top;  // with A the tree pass has formed r of the top nodes
  const int n_top = a.A ? 0 : a.n_top;
  auto node = [&](int i) { return a.A ? i : a.chain_node[i]; };
  const int G = (n_v + BS - 1) / BS, steps = G / 2 + 1;
  const long long per = lam_entries(n_v);
  const MT* lam = reinterpret_cast<const MT*>(a.lam);
  VT* delta = reinterpret_cast<VT*>(a.h);
  const bool one = a.lam_stride == 0;  // one matrix for all nodes
  const int cw = one || slots == 0 ? LW : slots;  // chain warps at work
  MT* slot = reinterpret_cast<MT*>(smem_raw) + (one ? 0 : (long long)warp * per);
  int q = (int)blockIdx.x * cw + warp;
  const int dq = (int)gridDim.x * cw;
  const bool chains = warp < cw && q < n_c;
  auto fetch = [&](int m) {  // lane 0: node m's matrix into this warp's slot
    mbar_expect_tx(&bar[warp], (uint32_t)(per * sizeof(MT)));
    bulk_g2s(slot, lam + m * a.lam_stride, (uint32_t)(per * sizeof(MT)), &bar[warp]);
  };
  if (slots > 0 && warp < cw && lane == 0) {
    mbar_init(&bar[warp], 1);
    fence_barrier_init();
    fence_proxy_async();
    if (one ? warp == 0 : chains) fetch(one ? 0 : node(q));
  }
  const bool mine = one ? warp == 0 : chains;  // a copy of this warp's is under way
  // the top warps: the first top node's sources into shared memory, its matrix towards the L2
  const int tid = (int)threadIdx.x - LW * 32;
  ST* part = reinterpret_cast<ST*>(smem_raw + round_up((size_t)slots * per * sizeof(MT), 128));  // ng n_v <= 256 sums
  VT* lsum = reinterpret_cast<VT*>(part + kWarps * 32);  // the warps' parts of delta
  const int2* src = reinterpret_cast<const int2*>(a.top_src);
  int s0 = 0, s1 = 0, m_top = 0;
  if (warp >= LW && (int)blockIdx.x < n_top) {
    m_top = a.top_nodes[blockIdx.x];
    s0 = a.top_src_off[blockIdx.x];
    s1 = a.top_src_off[blockIdx.x + 1];
    if (tid < min(kTopList, s1 - s0)) list[tid] = src[s0 + tid];
    const char* lm = reinterpret_cast<const char*>(lam + m_top * a.lam_stride);
    for (long long o = 128ll * tid; o < per * (long long)sizeof(MT); o += 128ll * 256)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(lm + o));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early_exit(a, nu, mode, flag, false)) {
    if (slots > 0 && mine) mbar_wait(&bar[warp], 0);  // the copy lands (bounded) before the CTA leaves
    return;
  }
  if (warp < LW) {
    if (one && slots > 0 && warp != 0 && !chains) return;
    uint32_t phase = 0;
    // ids are read two nodes ahead and r one node ahead of their use
    constexpr int RL = BS;  // 32 RL >= n_v
    const bool any = warp < cw && q < n_c;
    int m = any ? node(q) : 0, m1 = any && q + dq < n_c ? node(q + dq) : -1;
    VT rn[RL], sc = 1;
    auto read_r = [&](long long at) {
#pragma unroll
      for (int k = 0; k < RL; ++k) {
        const int j = lane + 32 * k;
        rn[k] = j < n_v ? reinterpret_cast<const VT*>(a.rpub)[at * n_v + j] : (VT)0;
      }
      if (a.pscale) sc = reinterpret_cast<const VT*>(a.pscale)[at];
    };
    if (any) read_r(m);
    for (; q < n_c && warp < cw; q += dq) {
      const int m2 = q + 2 * dq < n_c ? node(q + 2 * dq) : -1;
      const VT scale = sc;
#pragma unroll
      for (int k = 0; k < RL; ++k) rs[warp][lane + 32 * k] = rn[k];
      if (m1 >= 0) read_r(m1);
      if (slots > 0) {
        const bool ok = mbar_wait(one ? &bar[0] : &bar[warp], one ? 0 : phase, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
          if (lane == 0) a.flags[1] = SMPC_ETIMEOUT;
          mbar_wait(one ? &bar[0] : &bar[warp], one ? 0 : phase);  // bounded: let the copy land
          return;
        }
        phase ^= 1;
      }
      __syncwarp();
      VT acc[BS] = {};
      lam_steps<VT, BS>(slots > 0 ? slot : lam + m * a.lam_stride, G, rs[warp], 0, steps, acc);
      __syncwarp();  // the slot and r have been read
      if (slots > 0 && !one && lane == 0 && m1 >= 0) {
        fence_proxy_async();
        fetch(m1);
      }
      if (lane < G) {
#pragma unroll
        for (int c = 0; c < BS; ++c)
          if (BS * lane + c < n_v) delta[(long long)m * n_v + BS * lane + c] = acc[c] * scale;
      }
      m = m1;
      m1 = m2;
    }
    if (one && slots > 0 && warp == 0) mbar_wait(&bar[0], 0);  // bounded: also where it had no node
    return;
  }
  // a top node: r = the sum of its sources' two terms.  These are sums of many terms that
  // nearly cancel, and they move every scenario below: float32 ones run in the state type (two
  // float32), else the duals of the top nodes drift (plain sums over the chains: errors 3 to 8
  // times those of sums along the tree).
  const int tw = warp - LW;
  VT* rt = rs[LW];
  const VT* rp = reinterpret_cast<const VT*>(a.rpub);
  const VT* wb = reinterpret_cast<const VT*>(a.wbuf);
  for (int t = blockIdx.x; t < n_top; t += gridDim.x) {
    const bool first = t == (int)blockIdx.x;
    if (!first) {
      m_top = a.top_nodes[t];
      s0 = a.top_src_off[t];
      s1 = a.top_src_off[t + 1];
    }
    const long long m = m_top;
    // with 2 ng <= 8 warps a group of threads takes one column of every ng-th source, eight
    // sources (sixteen loads) in flight; the ids go through shared memory, kTopList at a time
    const int gw = (n_v + 31) / 32, ng = kWarps / gw, grp = tid / (32 * gw), j = tid - grp * 32 * gw;
    const bool on = grp < ng && j < n_v;
    ST sum = st_from<ST>(0.0);
    for (int i0 = s0; i0 < s1; i0 += kTopList) {
      const int cnt = min(kTopList, s1 - i0);
      if (!first || i0 > s0) {
        bar_top();  // the previous list has been used
        if (tid < cnt) list[tid] = src[i0 + tid];
        bar_top();
      }
      constexpr int B = 8;
      if (on)
        for (int i = grp; i < cnt; i += B * ng) {
          VT v[B], w[B];
#pragma unroll
          for (int k = 0; k < B; ++k) {  // behind the end: the last source again, not added
            const long long id = list[min(i + k * ng, cnt - 1)].x;
            v[k] = rp[id * n_v + j];
            w[k] = wb[id * n_k + j];
          }
#pragma unroll
          for (int k = 0; k < B; ++k)
            if (i + k * ng < cnt) {
              st_fma_acc(sum, (VT)1, v[k]);
              st_fma_acc(sum, (VT)list[i + k * ng].y, w[k]);
            }
        }
    }
    if (on) part[grp * n_v + j] = sum;
    bar_top();
    if (tid < 32 * BS) {
      ST v = st_from<ST>(0.0);
      if (tid < n_v) {
        v = part[tid];
        for (int g = 1; g < ng; ++g) v = st_add(v, part[g * n_v + tid]);
      }
      rt[tid] = st_val(v);
    }
    bar_top();
    // the steps shared by the warps, their sums added in order
    const int k0 = steps * tw / kWarps, k1 = steps * (tw + 1) / kWarps;
    VT acc[BS] = {};
    if (k0 < k1) lam_steps<VT, BS>(lam + m * a.lam_stride, G, rt, k0, k1, acc);
    if (lane < G) {
#pragma unroll
      for (int c = 0; c < BS; ++c) lsum[tw * (32 * BS) + BS * lane + c] = acc[c];
    }
    bar_top();
    const VT sc = a.pscale ? reinterpret_cast<const VT*>(a.pscale)[m] : (VT)1;
    for (int j = tid; j < n_v; j += 256) {
      VT v = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += lsum[w * (32 * BS) + j];
      delta[m * n_v + j] = v * sc;
    }
    // part is rewritten behind the next top node's first barrier, lsum behind later ones
  }
}
