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
//   lambda_apply  delta_n = Lambda_n r_n, one warp per chain node; one CTA per top node, which
//                 first forms its r from the chain heads and top nodes below it.  A top node's
//                 s and r are weighted sums over them (a head's xi counts once for every top
//                 node between the two), so no top node waits for another one.
// Per iteration on GB300, one pack per node (the launches of schedules 2 to 4 before): 2081
// nodes 39.5 us in float32 (104), 162 us in float64 (381); 21 111 nodes 191 us (577); one pack
// for all of 21 111 nodes 157 us (396).
// Vectors between the launches: h holds delta (n x n_v), rpub r of the chain nodes, spub s of
// the chain heads, wbuf w of the top nodes.

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
template <typename VT, typename P, typename F>
__device__ __forceinline__ void sparse_rows(const SpEnt<VT>* ent, const int* ptr, const int* id, int rows, const VT* X,
                                            int xs, int r0, int r1, P&& pre, F&& put) {
  constexpr int NB = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rw = (rows + 31) / 32, ng = (r1 - r0 + NB - 1) / NB;
  for (int task = warp; task < rw * ng; task += kWarps) {
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

template <typename VT>
__host__ __device__ inline size_t sweep_smem_bytes(int nnz, int depth, int n_x, int n_u, int n_v) {
  const int n_k = n_x + n_u;
  size_t b = sp_bytes<VT>(nnz, n_k, n_v);
  b += (size_t)(3 * n_x + 2 * n_u + (depth + 3) * (n_v + n_k)) * sizeof(VT);
  return round_up(b + (size_t)depth * sizeof(int), 16);
}

// Prox, dual update and w of node m on one warp (App. C; the arithmetic of
// Kern::warp_prox_staged).  z holds x and u on entry and w on return.  All of the node's
// loads are issued before the first use: lane l owns the tanks l + 32 k and the inputs
// l + 32 k, NT and NU of them at most.
template <typename VT, int NT, int NU>
__device__ __forceinline__ void sweep_prox(const IterArgs& a, int m, VT* z, const VT* bnd, int nu, VT& rmax, VT& hmax,
                                           VT& tmax) {
  using ST = typename St<VT>::T;
  const int lane = threadIdx.x & 31, n_x = a.n_x, n_u = a.n_u, nd = 2 * n_x + n_u, it = nu - 1;
  const VT *xs = bnd, *xhi = xs + n_x, *xlo = xhi + n_x, *uhi = xlo + n_x, *ulo = uhi + n_u;
  const ST* y1 = reinterpret_cast<const ST*>((it & 1) ? a.ybuf1 : a.ybuf0) + (long long)m * nd;
  ST* y2 = reinterpret_cast<ST*>((it & 1) ? a.ybuf0 : a.ybuf1) + (long long)m * nd;
  const VT* step_p = reinterpret_cast<const VT*>(a.step_p) + (long long)m * n_u;
  const VT* inv_p = reinterpret_cast<const VT*>(a.inv_p) + (long long)m * n_u;
  const ST zero = st_from<ST>(0.0);
  ST v1[NT], ws[NT], w1[NT], wz[NT], p1[NU], p2[NU];
  VT lp[NU], ip[NU];
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
#pragma unroll
  for (int k = 0; k < NU; ++k) {
    const int i = lane + 32 * k;
    p1[k] = p2[k] = zero;
    lp[k] = ip[k] = 1;
    if (i < n_u) {
      p1[k] = ld_state(y1 + 2 * n_x + i);
      p2[k] = ld_state(y2 + 2 * n_x + i);
      lp[k] = step_p[i];
      ip[k] = inv_p[i];
    }
  }
  const VT c = (VT)a.cvec[it], cn = (VT)a.cvec[it + 1];
  const VT ls = reinterpret_cast<const VT*>(a.step_s)[m], lz = reinterpret_cast<const VT*>(a.step_z)[m];
  const VT is = reinterpret_cast<const VT*>(a.inv_s)[m], iz = reinterpret_cast<const VT*>(a.inv_z)[m];
  const VT mus = reinterpret_cast<const VT*>(a.mu_s)[m], muz = (VT)a.gamma_d;
  const VT th = a.xbar && it > 0 ? (VT)a.theta[it] : (VT)1;  // ergodic average (theta_0 = 1)
  VT* xo = reinterpret_cast<VT*>(a.xout) + (long long)m * n_x;
  VT* uo = reinterpret_cast<VT*>(a.uout) + (long long)m * n_u;
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
      qs[k] = st_neg(q) ? q : zero;  // C = {x >= x_s}
      qz[k] = box_lr(st_axpy(wz[k], lz, x - xhi[e]), st_axpy(wz[k], lz, x - xlo[e]));
      const VT rs = st_val(qs[k]), rz = st_val(qz[k]);
      ps += rs * rs;
      pz += rz * rz;
    }
  }
  // the input blocks do not need the norms: they fill the reduction's latency
  VT rm = 0, hm = 0, tm = 0;
  bool bad = false;
#pragma unroll
  for (int k = 0; k < NU; ++k) {
    const int i = lane + 32 * k;
    if (i < n_u) {
      const VT u = z[n_x + i];
      const ST wp = st_extrap(p1[k], p2[k], c);
      const ST ypn = box_lr(st_axpy(wp, lp[k], u - uhi[i]), st_axpy(wp, lp[k], u - ulo[i]));
      const VT ep = st_val(st_sub(ypn, wp)) * ip[k];
      st_state(y2 + 2 * n_x + i, ypn);
      uo[i] = u;
      z[n_x + i] = st_extrap_val(ypn, p1[k], cn);
      if (a.ubar) {
        VT* b = reinterpret_cast<VT*>(a.ubar) + (long long)m * n_u + i;
        *b = it == 0 ? u : (VT)(((VT)1 - th) * *b + th * u);
      }
      rm = fmax(rm, fabs(ep));
      hm = fmax(hm, fabs(u));
      tm = fmax(tm, fabs(u - ep));
      bad |= !isfinite(st_val(ypn)) || !isfinite(u);
    }
  }
  ps = warp_sum(ps);
  pz = warp_sum(pz);
  const VT ds = sqrt(ps), dz = sqrt(pz);
  const VT ks = ds > mus ? mus / ds : (VT)1, kz = dz > muz ? muz / dz : (VT)1;
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const int e = lane + 32 * k;
    if (e < n_x) {
      const VT x = z[e];
      const ST ysn = st_scale(qs[k], ks), yzn = st_scale(qz[k], kz);
      const VT es = st_val(st_sub(ysn, ws[k])) * is, ez = st_val(st_sub(yzn, wz[k])) * iz;
      st_state(y2 + e, ysn);
      st_state(y2 + n_x + e, yzn);
      xo[e] = x;
      z[e] = st_extrap_val(ysn, v1[k], cn) + st_extrap_val(yzn, w1[k], cn);
      if (a.xbar) {
        VT* b = reinterpret_cast<VT*>(a.xbar) + (long long)m * n_x + e;
        *b = it == 0 ? x : (VT)(((VT)1 - th) * *b + th * x);
      }
      rm = fmax(rm, fmax(fabs(es), fabs(ez)));
      hm = fmax(hm, fabs(x));
      tm = fmax(tm, fmax(fabs(x - es), fabs(x - ez)));
      // the prox maps a non-finite v to 0, so the primal iterate is checked as well
      bad |= !isfinite(st_val(ysn)) || !isfinite(st_val(yzn)) || !isfinite(x);
    }
  }
  if (bad) a.flags[1] = SMPC_EDIVERGED;
  rmax = fmax(rmax, rm);
  hmax = fmax(hmax, hm);
  tmax = fmax(tmax, tm);
}

template <typename VT, int NT, int NU>
__global__ void __launch_bounds__(kThreads, NT == 8 ? 1 : sizeof(VT) == 4 ? 3 : 2)
    tree_sweep(const __grid_constant__ IterArgs a, int nu, int mode) {
  using ST = typename St<VT>::T;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int flag[2];
  __shared__ VT red[3 * kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_x = a.n_x, n_u = a.n_u, n_k = a.n_k, n_v = a.n_v, nnz = a.sp_nnz;
  // ---- constants of the factor and the tree, read while the previous launch drains
  const int blob = sp_bytes<VT>(nnz, n_k, n_v);
  for (int q = tid; q < blob / 16; q += kThreads)
    reinterpret_cast<uint4*>(smem_raw)[q] = reinterpret_cast<const uint4*>(a.sp)[q];
  const SpEnt<VT>* ek = reinterpret_cast<const SpEnt<VT>*>(smem_raw);
  const SpEnt<VT>* et = ek + nnz;
  const int* rptr = reinterpret_cast<const int*>(et + nnz);
  const int *rid = rptr + n_k + 1, *cptr = rid + n_k, *cid = cptr + n_v + 1;
  VT* bnd = reinterpret_cast<VT*>(smem_raw + blob);
  VT* V = bnd + 3 * n_x + 2 * n_u;  // delta, then v, then g and r: a row of n_v per node
  VT* Z = V + (a.depth + 3) * n_v;  // [Bbar; L] v, then x and u, then w and s: a row of n_k per node
  int* sid = reinterpret_cast<int*>(Z + (a.depth + 3) * n_k);
  for (int q = tid; q < 3 * n_x + 2 * n_u; q += kThreads) {
    const void* src = q < n_x ? a.x_s : q < 2 * n_x ? a.x_max : q < 3 * n_x ? a.x_min : q < 3 * n_x + n_u ? a.u_max : a.u_min;
    const int i = q < 3 * n_x ? q % n_x : (q - 3 * n_x) % n_u;
    bnd[q] = reinterpret_cast<const VT*>(src)[i];
  }
  // chains first (the long tasks), then the top nodes
  const int b = (int)blockIdx.x < a.n_chains ? a.n_top + blockIdx.x : blockIdx.x - a.n_chains;
  const int4 d0 = *reinterpret_cast<const int4*>(a.seg + (long long)kSegInts * b);
  const int4 d1 = *reinterpret_cast<const int4*>(a.seg + (long long)kSegInts * b + 4);
  const int pl = d0.z, len = d1.y, tree = d0.w;
  const int L = pl + len;                   // the path (root .. parent), then the segment's own nodes
  const int own = len == 0 ? pl - 1 : pl;   // first own row (a top node ends its path)
  for (int r = tid; r < L; r += kThreads) sid[r] = r < pl ? a.path_node[d0.y + r] : a.chain_node[d1.x + r - pl];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early_exit(a, nu, mode, flag, true)) return;  // its barrier publishes the above
  const bool prox = (mode & MODE_PROX) != 0 && nu >= 1;
  if (!tree_active(a, tree, nu)) return;  // a forest's tree that stopped keeps its iterates
  VT rmax = 0, hmax = 0, tmax = 0;
  if (prox) {
    const VT* delta = reinterpret_cast<const VT*>(a.h);
    for (int r = warp; r < L; r += kWarps) {
      const VT* src = delta + (long long)sid[r] * n_v;
      for (int j = lane; j < n_v; j += 32) V[r * n_v + j] = src[j];
    }
    __syncthreads();
    if (tid < n_v) {  // v along the path
      VT v = 0;
#pragma unroll 8
      for (int r = 0; r < L; ++r) V[r * n_v + tid] = v += V[r * n_v + tid];
    }
    __syncthreads();
    const VT* E = reinterpret_cast<const VT*>(a.e);
    const VT* UH = reinterpret_cast<const VT*>(a.uhat);
    sparse_rows<VT>(
        ek, rptr, rid, n_k, V, n_v, 0, L,
        [&](int r, int e) -> VT {
          const long long m = sid[r];
          return e < n_x ? E[m * n_x + e] : r >= own ? UH[m * n_u + e - n_x] : (VT)0;
        },
        [&](int r, int e, VT v) { Z[r * n_k + e] = v; });
    __syncthreads();
    if (tid < n_x) {  // x_n = x_parent + Bbar v_n + e_n
      VT x = reinterpret_cast<const VT*>(a.p0)[(long long)tree * n_x + tid];
#pragma unroll 8
      for (int r = 0; r < L; ++r) Z[r * n_k + tid] = x += Z[r * n_k + tid];
    }
    __syncthreads();
    for (int r = own + warp; r < L; r += kWarps)
      sweep_prox<VT, NT, NU>(a, sid[r], Z + r * n_k, bnd, nu, rmax, hmax, tmax);
  } else {  // w^nu without a prox: the first iteration
    const VT c = (VT)a.cvec[nu];
    const int nd = 2 * n_x + n_u;
    for (int r = own + warp; r < L; r += kWarps) {
      const ST* ya = reinterpret_cast<const ST*>((nu & 1) ? a.ybuf1 : a.ybuf0) + (long long)sid[r] * nd;
      const ST* yb = reinterpret_cast<const ST*>((nu & 1) ? a.ybuf0 : a.ybuf1) + (long long)sid[r] * nd;
      for (int e = lane; e < n_k; e += 32) {
        if (e < n_x)
          Z[r * n_k + e] = st_val(st_add(st_extrap(ld_state(ya + e), ld_state(yb + e), c),
                                         st_extrap(ld_state(ya + n_x + e), ld_state(yb + n_x + e), c)));
        else
          Z[r * n_k + e] = st_val(st_extrap(ld_state(ya + n_x + e), ld_state(yb + n_x + e), c));
      }
    }
  }
  if (prox) {  // residual maxima (Sec. IV-E)
    rmax = warp_max(rmax);
    hmax = warp_max(hmax);
    tmax = warp_max(tmax);
    if (lane == 0) {
      red[warp] = rmax;
      red[kWarps + warp] = hmax;
      red[2 * kWarps + warp] = tmax;
    }
  }
  __syncthreads();
  if (prox && tid < 3) {
    VT v = 0;
    for (int w = 0; w < kWarps; ++w) v = fmax(v, red[tid * kWarps + w]);
    atomic_max_nonneg(a.res + 3ll * (nu - 1) + tid, (double)v);
    if (a.res_tree) atomic_max_nonneg(a.res_tree + 3ll * ((long long)(nu - 1) * a.R + tree) + tid, (double)v);
  }
  if (!(mode & MODE_BWD)) return;
  if (len == 0) {  // a top node: its w, for lambda_apply
    VT* w = reinterpret_cast<VT*>(a.wbuf) + (long long)sid[own] * n_k;
    for (int e = tid; e < n_k; e += kThreads) w[e] = Z[own * n_k + e];
    return;
  }
  if (tid < n_x) {  // s along the chain, bottom-up
    VT s = 0;
#pragma unroll 8
    for (int r = L - 1; r >= own; --r) Z[r * n_k + tid] = s += Z[r * n_k + tid];
    reinterpret_cast<VT*>(a.spub)[(long long)sid[own] * n_x + tid] = s;
  }
  __syncthreads();
  const VT* beta = reinterpret_cast<const VT*>(a.beta);
  sparse_rows<VT>(
      et, cptr, cid, n_v, Z, n_k, own, L, [&](int r, int j) -> VT { return beta[(long long)sid[r] * n_v + j]; },
      [&](int r, int j, VT v) { V[r * n_v + j] = v; });
  __syncthreads();
  if (tid < n_v) {  // r along the chain
    VT* R = reinterpret_cast<VT*>(a.rpub);
    VT s = 0;
#pragma unroll 8
    for (int r = L - 1; r >= own; --r) {
      s += V[r * n_v + tid];
      R[(long long)sid[r] * n_v + tid] = s;
    }
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

// Steps [k0, k1) of one matrix on a warp: acc += the part of Lambda r in row block `lane`.
// rs: r, zero-padded to G BS entries, 16-byte aligned.
template <typename VT, int BS>
__device__ __forceinline__ void lam_steps(const VT* lam, int G, const VT* rs, int k0, int k1, VT (&acc)[BS]) {
  constexpr int CE = 16 / (int)sizeof(VT), NC = BS * BS / CE;
  constexpr int U = BS == 8 ? 1 : sizeof(VT) == 4 ? 4 : 2;  // steps whose loads are in flight together
  const int lane = threadIdx.x & 31;
  const int I = lane < G ? lane : 0;  // idle lanes repeat lane 0's loads; nothing of theirs is used
  VT ri[BS], tr[BS];
#pragma unroll
  for (int r = 0; r < BS; ++r) {
    ri[r] = rs[BS * I + r];
    tr[r] = 0;
  }
  const int from = I + 1 < G ? I + 1 : 0;
  for (int kb = k0; kb < k1; kb += U) {
    VT A[U][BS * BS];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = min(kb + u, k1 - 1);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        VT t[CE];
        ld16(lam + ((long long)(k * NC + c) * G + I) * CE, t);
#pragma unroll
        for (int q = 0; q < CE; ++q) A[u][c * CE + q] = t[q];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = kb + u;
      if (k >= k1) break;
      int J = I + k;
      if (J >= G) J -= G;
      const VT* rj = rs + BS * J;
#pragma unroll
      for (int q = 0; q < BS; ++q) tr[q] = __shfl_sync(0xffffffffu, tr[q], from);
#pragma unroll
      for (int r = 0; r < BS; ++r)
#pragma unroll
        for (int q = 0; q < BS; ++q) {
          acc[r] += A[u][r * BS + q] * rj[q];
          if (k > 0) tr[q] += A[u][r * BS + q] * ri[r];
        }
    }
  }
  int back = (I - (k1 - 1)) % G;  // row block I's travelling sums are on lane I - (k1 - 1)
  if (back < 0) back += G;
#pragma unroll
  for (int q = 0; q < BS; ++q) acc[q] += __shfl_sync(0xffffffffu, tr[q], back);
}

// acc += w v, the product taken exactly
__device__ __forceinline__ void st_fma_acc(DS& acc, float w, float v) { acc = st_axpy(acc, w, v); }
__device__ __forceinline__ void st_fma_acc(double& acc, double w, double v) { acc = fma(w, v, acc); }

template <typename VT, int BS>
__global__ void __launch_bounds__(kThreads) lambda_apply(const __grid_constant__ IterArgs a, int nu, int mode) {
  using ST = typename St<VT>::T;
  grid_dep_sync();
  __shared__ int flag[2];
  __shared__ __align__(16) VT rs[kWarps][32 * BS];
  extern __shared__ __align__(128) unsigned char smem_raw[];
  if (early_exit(a, nu, mode, flag, false)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_x = a.n_x, n_k = a.n_k, n_v = a.n_v;
  const int G = (n_v + BS - 1) / BS, steps = G / 2 + 1;
  const VT* lam = reinterpret_cast<const VT*>(a.lam);
  VT* delta = reinterpret_cast<VT*>(a.h);
  if ((int)blockIdx.x >= a.n_top) {  // a warp per chain node
    const int q = ((int)blockIdx.x - a.n_top) * kWarps + warp;
    if (q >= a.n - a.n_top) return;
    const long long m = a.chain_node[q];
    const VT* r = reinterpret_cast<const VT*>(a.rpub) + m * n_v;
    for (int j = lane; j < 32 * BS; j += 32) rs[warp][j] = j < n_v ? r[j] : (VT)0;
    __syncwarp();
    VT acc[BS] = {};
    lam_steps<VT, BS>(lam + m * a.lam_stride, G, rs[warp], 0, steps, acc);
    const VT sc = a.pscale ? reinterpret_cast<const VT*>(a.pscale)[m] : (VT)1;
    if (lane < G) {
#pragma unroll
      for (int c = 0; c < BS; ++c)
        if (BS * lane + c < n_v) delta[m * n_v + BS * lane + c] = acc[c] * sc;
    }
    return;
  }
  // a top node: [S; P | R] = the weighted sums of s (weights: top nodes between), psi and r
  // (or beta) over the heads and top nodes below; then r = R + [Bbar; L]' [S; P].  These are
  // sums of hundreds of terms that nearly cancel, and they move every scenario below: float32
  // ones run in the state type (two float32), else the duals of the top nodes drift.
  const int W = n_k + n_v;
  ST* part = reinterpret_cast<ST*>(smem_raw);  // kWarps x W, in the state type (see above)
  const long long m = a.top_nodes[blockIdx.x];
  const VT* sp = reinterpret_cast<const VT*>(a.spub);
  const VT* rp = reinterpret_cast<const VT*>(a.rpub);
  const VT* wb = reinterpret_cast<const VT*>(a.wbuf);
  const VT* beta = reinterpret_cast<const VT*>(a.beta);
  const int h0 = a.top_src_off[2 * blockIdx.x], t0 = a.top_src_off[2 * blockIdx.x + 1],
            t1 = a.top_src_off[2 * blockIdx.x + 2];
  // a warp takes every kWarps-th source with all its columns in flight
  constexpr int NC = 8;  // 32 NC >= n_k, n_v
  const int2* src = reinterpret_cast<const int2*>(a.top_src);
  ST y[NC], g[NC];  // [S; P] and R, columns lane + 32 k
#pragma unroll
  for (int k = 0; k < NC; ++k) y[k] = g[k] = st_from<ST>(0.0);
#pragma unroll 4
  for (int q = h0 + warp; q < t0; q += kWarps) {
    const int2 s = src[q];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int e = lane + 32 * k;
      if (e < n_x) st_fma_acc(y[k], (VT)s.y, sp[(long long)s.x * n_x + e]);
      if (e < n_v) st_fma_acc(g[k], (VT)1, rp[(long long)s.x * n_v + e]);
    }
  }
#pragma unroll 2
  for (int q = t0 + warp; q < t1; q += kWarps) {
    const int2 s = src[q];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int e = lane + 32 * k;
      if (e < n_k) st_fma_acc(y[k], e < n_x ? (VT)s.y : (VT)1, wb[(long long)s.x * n_k + e]);
      if (e < n_v) st_fma_acc(g[k], (VT)1, beta[(long long)s.x * n_v + e]);
    }
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const int e = lane + 32 * k;
    if (e < n_k) part[warp * W + e] = y[k];
    if (e < n_v) part[warp * W + n_k + e] = g[k];
  }
  __syncthreads();
  for (int e = tid; e < W; e += kThreads) {
    ST v = part[e];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) v = st_add(v, part[w * W + e]);
    part[e] = v;  // entry e of every warp's row is read and written by this thread only
  }
  __syncthreads();
  const int nnz = a.sp_nnz;
  const SpEnt<VT>* et = reinterpret_cast<const SpEnt<VT>*>(a.sp) + nnz;
  const int* rptr = reinterpret_cast<const int*>(et + nnz);
  const int *cptr = rptr + 2 * n_k + 1, *cid = cptr + n_v + 1;
  for (int j = tid; j < 32 * BS; j += kThreads) {
    if (j < n_v) {
      const int col = cid[j];
      ST v = part[n_k + col];
      for (int q = cptr[j]; q < cptr[j + 1]; ++q) v = st_add(v, st_scale(part[et[q].c], et[q].v));
      rs[0][col] = st_val(v);
    } else {
      rs[0][j] = 0;
    }
  }
  __syncthreads();
  // the steps shared by the warps, their sums added in order
  const int k0 = steps * warp / kWarps, k1 = steps * (warp + 1) / kWarps;
  VT acc[BS] = {};
  if (k0 < k1) lam_steps<VT, BS>(lam + m * a.lam_stride, G, rs[0], k0, k1, acc);
  __syncthreads();  // part is free
  VT* lsum = reinterpret_cast<VT*>(smem_raw);
  if (lane < G) {
#pragma unroll
    for (int c = 0; c < BS; ++c) lsum[warp * (32 * BS) + BS * lane + c] = acc[c];
  }
  __syncthreads();
  const VT sc = a.pscale ? reinterpret_cast<const VT*>(a.pscale)[m] : (VT)1;
  for (int j = tid; j < n_v; j += kThreads) {
    VT v = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) v += lsum[w * (32 * BS) + j];
    delta[m * n_v + j] = v * sc;
  }
}
template <typename VT>
__host__ __device__ inline size_t lambda_smem_bytes(int n_k, int n_v) {
  const int W = n_k + n_v, R = 32 * lam_bs(n_v);
  return (size_t)kWarps * (W > R ? W : R) * kStateSize;
}
