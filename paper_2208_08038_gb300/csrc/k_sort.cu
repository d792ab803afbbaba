// k_sort.cu -- integer work: the counting sort of particles by tile-major cell
// (key = tile * cells_per_tile + cell within tile) as one cooperative kernel,
// which does its work only when the device status word says a particle left
// its tile's margin; the seeded device-side
// medium generator; and the FP64 Gauss-law residual.
#include <cstring>

#include "bp_internal.cuh"

namespace {

// blocks for n items; the kernels launched with it are grid-stride loops, so
// the cap (two waves of 256-thread blocks on 152 SMs) only bounds the grid
int blocks_for(long long n, int bs, long long cap = 152LL * 16) {
  long long b = (n + bs - 1) / bs;
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

__device__ __forceinline__ int sort_key(const GridP &g, int cell) {
  int cc[3];
  unpack_cell(g, cell, cc);
  const int c0 = cc[0], c1 = cc[1], c2 = cc[2];
  int t = c0 / g.L[0] + g.nt[0] * (c1 / g.L[1] + g.nt[1] * (c2 / g.L[2]));
  int l = c0 % g.L[0] + g.L[0] * (c1 % g.L[1] + g.L[1] * (c2 % g.L[2]));
  return t * g.cpt + l;
}

constexpr int SORT_BS = 512;

// exclusive scan over the block; total: the block's sum
__device__ __forceinline__ int block_exclusive_scan(int v, int *sh, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = lane < (blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    sh[lane] = w;
  }
  __syncthreads();
  int base = warp ? sh[warp - 1] : 0;
  total = sh[(blockDim.x >> 5) - 1];
  __syncthreads();
  return base + x - v;
}

// A barrier over the blocks of a cooperative launch (all resident at once).
// The wait is bounded (SortBufs::polls): false, with ST_TIMEOUT set, when it
// gives up.  The barrier, the histogram and the particle arrays are then
// left as they are, so every later sort and push stays away (status[2]) until
// the host has cleared the first two and the particles are loaded anew.
__device__ __forceinline__ bool grid_barrier(const SortBufs &b, int *status) {
  unsigned *const bar = b.bar;
  __shared__ int passed;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned *gen = bar + 1;
    const unsigned g0 = *gen;
    __threadfence();
    passed = 1;
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      bar[0] = 0u;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      passed = 0;
      for (int it = 0; it < b.polls; ++it) {
        if (*gen != g0) {
          passed = 1;
          break;
        }
        __nanosleep(64);
      }
      if (!passed) set_timeout(status);
    }
    __threadfence();
  }
  __syncthreads();
  return passed != 0;
}

// The counting sort by tile-major cell of the species that ask for it, as one
// cooperative kernel that returns at once unless the status word does (a
// particle left its tile's margin): count, scan (each block its share of the cells, the
// blocks' totals summed by every block), scatter to the scratch arrays, copy
// back and clear the histogram.  As a conditional graph node with the phases
// as nine launches a species the check alone took 14 to 21 us of every step
// (1D medium: step 35 us with the conditional node, 21 us without); an
// exiting launch takes 2 to 3.
struct SortArgs {
  int nsp;
  PartP p[BP_MAX_SPECIES];
  int two[BP_MAX_SPECIES];
  SortBufs b;
  int *status;
};
__global__ void __launch_bounds__(SORT_BS, 3) k_sort(const __grid_constant__ GridP g, const __grid_constant__ SortArgs S) {
  // every block has read the flag when the last barrier lets one clear it
  const int4 st = __ldcv(reinterpret_cast<const int4 *>(S.status));
  if (!(st.x & ST_NEED_SORT) || st.z) return;
  const int which = st.y;  // bit s: species s; 0: all
  __shared__ int sh[32];
  const long long nh = g.ncell + 1;
  const long long tid = blockIdx.x * (long long)SORT_BS + threadIdx.x, nth = (long long)gridDim.x * SORT_BS;
  int *const hist = S.b.hist, *const bsum = S.b.bsum;
  const long long per = ((nh + gridDim.x - 1) / gridDim.x + SORT_BS - 1) / SORT_BS * SORT_BS;
  const long long h0 = (long long)blockIdx.x * per, h1 = h0 + per < nh ? h0 + per : nh;
  for (int s = 0; s < S.nsp; ++s) {
    if (which && !(which >> s & 1)) continue;
    const PartP p = S.p[s];
    const long long cap = p.cap;
    const int n = p.tstart[g.ntiles];
    // (the histogram is kept clear between sorts)
    for (long long q = tid; q < n; q += nth) {
      const int c = p.cell[q];
      if (c >= 0) atomicAdd(hist + sort_key(g, c), 1);
    }
    if (!grid_barrier(S.b, S.status)) return;
    int sum = 0, total;
    for (long long q = h0 + threadIdx.x; q < h1; q += SORT_BS) sum += hist[q];
    block_exclusive_scan(sum, sh, total);
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
    if (!grid_barrier(S.b, S.status)) return;
    int carry = 0;
    sum = 0;
    for (int q = threadIdx.x; q < (int)blockIdx.x; q += SORT_BS) sum += bsum[q];
    block_exclusive_scan(sum, sh, carry);
    for (long long q = h0; q < h1; q += SORT_BS) {
      const long long k = q + threadIdx.x;
      const int v = k < h1 ? hist[k] : 0;
      const int ex = carry + block_exclusive_scan(v, sh, total);
      if (k < h1) {
        hist[k] = ex;
        // the tile ranges; entry ncell is the count
        if (k % g.cpt == 0) p.tstart[k / g.cpt] = ex;
      }
      carry += total;
    }
    if (!grid_barrier(S.b, S.status)) return;
    for (long long q = tid; q < n; q += nth) {
      const int c = p.cell[q];
      if (c < 0) continue;
      const int dst = atomicAdd(hist + sort_key(g, c), 1);
      if (dst < 0 || dst >= cap) {  // only if the histogram was not clear
        atomicOr(S.status, ST_DOMAIN);
        continue;
      }
      float *tf = S.b.tmp_f + dst;
      S.b.tmp_cell[dst] = c;
      for (int a = 0; a < g.D; ++a, tf += cap) *tf = p.off[a * cap + q];
      for (int a = 0; a < 3; ++a, tf += cap) *tf = p.u1[a * cap + q];
      if (S.two[s]) {
        for (int a = 0; a < 3; ++a, tf += cap) *tf = p.r[a * cap + q];
        for (int a = 0; a < 3; ++a, tf += cap) *tf = p.u2[a * cap + q];
      }
      S.b.tmp_i[dst] = p.id[q];
      if (p.pidx) S.b.tmp_i[cap + dst] = p.pidx[q];
    }
    if (!grid_barrier(S.b, S.status)) return;
    const int m = p.tstart[g.ntiles];
    for (long long q = tid; q < nh; q += nth) hist[q] = 0;
    for (long long q = tid; q < m; q += nth) {
      const float *tf = S.b.tmp_f + q;
      p.cell[q] = S.b.tmp_cell[q];
      for (int a = 0; a < g.D; ++a, tf += cap) p.off[a * cap + q] = *tf;
      for (int a = 0; a < 3; ++a, tf += cap) p.u1[a * cap + q] = *tf;
      if (S.two[s]) {
        for (int a = 0; a < 3; ++a, tf += cap) p.r[a * cap + q] = *tf;
        for (int a = 0; a < 3; ++a, tf += cap) p.u2[a * cap + q] = *tf;
      }
      p.id[q] = S.b.tmp_i[q];
      if (p.pidx) p.pidx[q] = S.b.tmp_i[cap + q];
    }
    if (!grid_barrier(S.b, S.status)) return;
  }
  if (tid == 0) {
    S.status[1] = 0;
    if (st.w) S.status[3] = 0;  // a load's sort: the species it did not see are still to be sorted
    else atomicAnd(S.status, ~ST_NEED_SORT);
  }
}

// every species of the next launch_sort, a load's, is to be sorted
__global__ void k_set_flag(int *status) {
  if (status[0] & ST_NEED_SORT) status[3] = 1;
  status[1] = 0;
  status[0] |= ST_NEED_SORT;
}

// the status word cleared for a load, and what it held of other species' need
// set again after a load that failed
__global__ void k_load_begin(int *status) {
  if (status[0] & ST_NEED_SORT) status[3] = 1;
  status[0] = 0;
}
__global__ void k_load_failed(int *status) {
  if (status[3]) status[0] |= ST_NEED_SORT;
  status[1] = status[3] = 0;
}

// ---------------------------------------------------------------------------
// device medium: ion g = cell rank * ppc + p over the cell box [lo, hi);
// position x_a = (c_a + U(3g + a)) dx_a, momentum sigma N(3g + a); the
// two bodies start together (r = 0) with u1 = u2 = u_c for neutral ions and
// the non-relativistic split of p1 + p2 = p_c, q1 v1 + q2 v2 = 0 otherwise

__global__ void k_gen_medium(GridP g, SpecP sp, PartP p, int lo0, int lo1, int lo2, int e0, int e1, int ppc,
                             uint64_t kpos, uint64_t kmom, double sigma, long long first, long long count,
                             long long out0) {
  const long long cap = p.cap;
  const int lo[3] = {lo0, lo1, lo2}, ext[3] = {e0, e1, 1};
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < count;
       q += (long long)gridDim.x * blockDim.x) {
    long long gi = first + q;
    long long rem = gi / ppc;
    int cell[3] = {0, 0, 0};
    float off[3] = {0.0f, 0.0f, 0.0f};
    for (int a = 0; a < g.D; ++a) {
      long long e = a < 2 ? ext[a] : rem + 1;
      int ca = (int)(a < g.D - 1 ? rem % e : rem) + lo[a];
      if (a < g.D - 1) rem /= e;
      double u = sm64_uniform(kpos, (uint64_t)(3 * gi + a));
      double x = ((double)ca + u) * g.dxd[a];
      double X = x / g.dxd[a];
      double fl = floor(X);
      float f = (float)(X - fl);
      int ci = (int)fl;
      if (f >= 1.0f) { f = 0.0f; ci += 1; }
      if (ci >= g.n[a]) {
        // the offset of an ion at the very end of the grid's last cell rounds
        // up to 1 (one position in 2^25): a periodic axis wraps, on an open
        // one the ion stays in the cell (cell n would index past the grid)
        if (g.bc[a] == BP_PERIODIC) {
          ci = 0;
        } else {
          ci = g.n[a] - 1;
          f = 0.99999994f;
        }
      }
      cell[a] = ci;
      off[a] = f;
    }
    double uc[3] = {0.0, 0.0, 0.0};
    if (sigma > 0) {
      for (int a = 0; a < 3; ++a) {
        uint64_t c = (uint64_t)(3 * gi + a);
        double u1 = sm64_uniform(kmom, 2 * c), u2 = sm64_uniform(kmom, 2 * c + 1);
        uc[a] = sigma * sqrt(-2.0 * log(1.0 - u1)) * cos(6.283185307179586476925 * u2);
      }
    }
    long long o = out0 + q;
    p.cell[o] = pack_cell(g, cell[0], cell[1], cell[2]);
    for (int a = 0; a < g.D; ++a) p.off[a * cap + o] = off[a];
    if (sp.kind == BP_TWO_BODY) {
      double qc = sp.q1d + sp.q2d;
      for (int a = 0; a < 3; ++a) {
        double u1, u2;
        if (qc == 0.0) {
          u1 = u2 = uc[a];
        } else {
          u1 = (sp.m1d + sp.m2d) * uc[a] / (sp.m1d - sp.m2d * sp.q1d / sp.q2d);
          u2 = -sp.q1d * u1 / sp.q2d;
        }
        p.u1[a * cap + o] = (float)u1;
        p.u2[a * cap + o] = (float)u2;
        p.r[a * cap + o] = 0.0f;
      }
    } else {
      for (int a = 0; a < 3; ++a) p.u1[a * cap + o] = (float)uc[a];
    }
    p.id[o] = (int)gi;
    if (p.pidx) p.pidx[o] = 0;
  }
}

// ---------------------------------------------------------------------------
// FP64 Gauss-law residual: rho from the stored positions (quadratic shape at
// nodes), then R = div E - rho

__global__ void k_rho(GridP g, SpecP sp, PartP p, double *rho) {
  const long long cap = p.cap;
  const int n = p.tstart[g.ntiles];
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    int cell = p.cell[q];
    if (cell < 0) continue;
    int c[3];
    unpack_cell(g, cell, c);
    const int nb = sp.kind == BP_TWO_BODY ? 2 : 1;
    for (int b = 0; b < nb; ++b) {
      double qw = (b == 0 ? sp.q1d : sp.q2d) * sp.wd;
      int base[3], cnt[3];
      double w[3][3];
      for (int a = 0; a < 3; ++a) {
        if (a >= g.D) {
          base[a] = 0;
          cnt[a] = 1;
          w[a][0] = 1.0;
          continue;
        }
        double X = (double)c[a] + (double)p.off[a * cap + q];
        if (b == 1) X -= (double)p.r[a * cap + q] / g.dxd[a];
        double nn = floor(X + 0.5);
        double xi = X - nn;
        base[a] = (int)nn - 1;
        cnt[a] = 3;
        w[a][0] = 0.5 * (0.5 - xi) * (0.5 - xi);
        w[a][1] = 0.75 - xi * xi;
        w[a][2] = 0.5 * (0.5 + xi) * (0.5 + xi);
      }
      for (int kk = 0; kk < cnt[2]; ++kk)
        for (int jj = 0; jj < cnt[1]; ++jj)
          for (int ii = 0; ii < cnt[0]; ++ii) {
            int x[3] = {base[0] + ii, base[1] + jj, base[2] + kk};
            bool ok = true;
            for (int a = 0; a < g.D; ++a) {
              if (g.bc[a] == BP_PERIODIC) x[a] = wrap_mod(x[a], g.n[a]);
              else ok &= x[a] >= 0 && x[a] < g.n[a];
            }
            if (!ok) continue;
            long long id = x[0] + (long long)g.n[0] * (x[1] + (long long)g.n[1] * x[2]);
            atomicAdd(rho + id, qw * w[0][ii] * w[1][jj] * w[2][kk]);
          }
    }
  }
}

__global__ void k_divE(GridP g, const float *Ex, const float *Ey, const float *Ez, double *R) {
  const float *E[3] = {Ex, Ey, Ez};
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < g.ncell;
       q += (long long)gridDim.x * blockDim.x) {
    int c[3] = {(int)(q % g.n[0]), (int)((q / g.n[0]) % g.n[1]), (int)(q / ((long long)g.n[0] * g.n[1]))};
    double div = 0.0;
    for (int a = 0; a < g.D; ++a) {
      int x[3] = {c[0], c[1], c[2]};
      x[a] -= 1;
      double lo = 0.0;
      if (g.bc[a] == BP_PERIODIC) x[a] = wrap_mod(x[a], g.n[a]);
      if (x[a] >= 0) lo = (double)E[a][x[0] + (long long)g.n[0] * (x[1] + (long long)g.n[1] * x[2])];
      div += ((double)E[a][q] - lo) / g.dxd[a];
    }
    R[q] = div - R[q];
  }
}


// ---------------------------------------------------------------------------
// load: FP64 ion positions / momenta (caller's layout, staged on the device)
// to the particle arrays.  Initial conditions of Sec. 2: both bodies at the
// ion position (r = 0); u1 = u2 = u_c for neutral ions, else the
// non-relativistic solution of p1 + p2 = p_c, q1 v1 + q2 v2 = 0.

__global__ void k_load_convert(GridP g, SpecP sp, PartP p, const double *x, const double *u, const int *pidx,
                               long long first, long long count, int *status) {
  const long long cap = p.cap;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < count;
       q += (long long)gridDim.x * blockDim.x) {
    const long long o = first + q;
    int cell[3] = {0, 0, 0};
    bool bad = false, nonfinite = false;
    for (int a = 0; a < g.D; ++a) {
      double xa = x[q * g.D + a];
      nonfinite |= !isfinite(xa);
      double X = xa / g.dxd[a];
      double fl = floor(X);
      float f = (float)(X - fl);
      long long ci = (long long)fl;
      if (f >= 1.0f) { f = 0.0f; ci += 1; }
      if (g.bc[a] == BP_PERIODIC) {
        long long m = ci % g.n[a];
        ci = m < 0 ? m + g.n[a] : m;
      } else if (ci < 0 || ci >= g.n[a]) {
        bad = true;
        ci = 0;
      }
      cell[a] = (int)ci;
      p.off[a * cap + o] = f;
    }
    int pi = 0;
    if (pidx) {
      pi = pidx[q];
      if (pi < 0 || (sp.kind == BP_TWO_BODY && pi >= sp.nac)) { bad = true; pi = 0; }
      p.pidx[o] = pi;
    }
    for (int a = 0; a < 3; ++a) {
      double uc = u ? u[q * 3 + a] : 0.0;
      nonfinite |= !isfinite(uc);
      if (sp.kind != BP_TWO_BODY) {
        p.u1[a * cap + o] = (float)uc;
      } else {
        double u1, u2;
        if (sp.q1d + sp.q2d == 0.0) {
          u1 = u2 = uc;
        } else {
          u1 = (sp.m1d + sp.m2d) * uc / (sp.m1d - sp.m2d * sp.q1d / sp.q2d);
          u2 = -sp.q1d * u1 / sp.q2d;
        }
        p.u1[a * cap + o] = (float)u1;
        p.u2[a * cap + o] = (float)u2;
        p.r[a * cap + o] = 0.0f;
      }
    }
    p.cell[o] = (bad || nonfinite) ? -1 : pack_cell(g, cell[0], cell[1], cell[2]);
    p.id[o] = (int)o;
    if (bad) atomicOr(status, ST_DOMAIN);
    if (nonfinite) atomicOr(status, ST_NONFINITE);
  }
}

}  // namespace

int sort_blocks(int sms) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sort, SORT_BS, 0) != cudaSuccess || per < 1) return -1;
  return sms * per;
}

cudaError_t launch_sort(const GridP &g, int nsp, const SpecP *sp, const PartP *p, const SortBufs &b, int *status,
                        cudaStream_t s) {
  SortArgs S;
  memset(&S, 0, sizeof S);
  S.nsp = nsp;
  for (int k = 0; k < nsp; ++k) {
    S.p[k] = p[k];
    S.two[k] = sp[k].kind == BP_TWO_BODY;
  }
  S.b = b;
  S.status = status;
  // A block for every 4096 cells and particles, at least 16: the exit of an
  // unneeded sort and its barriers cost by the block (1D scan, 23.2 us a step
  // with all 456 resident blocks, 21.9 with 152), its phases gain by it (4.2 M
  // electrons: 495 and 528 us).
  long long work = g.ncell;
  for (int k = 0; k < nsp; ++k) work += p[k].cap;
  const long long want = work / 4096 < 16 ? 16 : work / 4096;
  const unsigned nb = (unsigned)(want < b.blocks ? want : b.blocks);
  void *args[2] = {(void *)&g, (void *)&S};
  return cudaLaunchCooperativeKernel((const void *)k_sort, dim3(nb), dim3(SORT_BS), args, 0, s);
}

void launch_set_sort_flag(int *status, cudaStream_t s) { k_set_flag<<<1, 1, 0, s>>>(status); }
void launch_load_begin(int *status, cudaStream_t s) { k_load_begin<<<1, 1, 0, s>>>(status); }
void launch_load_failed(int *status, cudaStream_t s) { k_load_failed<<<1, 1, 0, s>>>(status); }

// particles whose load id is in the sorted list sid[0..n): copy the raw
// state of particle slot i to row k of out (k = position of its id in the
// list): cell, then D offsets, r[3], u1[3], u2[3] as floats
__global__ void k_pick(PartP p, int D, int two, long long count, const int *sid, const int *srow, int n, int *cell_out,
                       float *out, unsigned char *found) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = p.cell[i];
    if (c < 0) continue;
    const int id = p.id[i];
    int lo = 0, hi = n;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sid[mid] < id) lo = mid + 1;
      else hi = mid;
    }
    if (lo >= n || sid[lo] != id) continue;
    const int k = srow[lo];
    cell_out[k] = c;
    float *o = out + (size_t)k * 12;
    for (int a = 0; a < D; ++a) o[a] = p.off[a * p.cap + i];
    for (int a = 0; a < 3; ++a) {
      o[3 + a] = two ? p.r[a * p.cap + i] : 0.0f;
      o[6 + a] = p.u1[a * p.cap + i];
      o[9 + a] = two ? p.u2[a * p.cap + i] : 0.0f;
    }
    found[k] = 1;
  }
}

void launch_pick(const PartP &p, int D, int two, long long count, const int *sid, const int *srow, int n,
                 int *cell_out, float *out, unsigned char *found, cudaStream_t s) {
  k_pick<<<blocks_for(count, 256), 256, 0, s>>>(p, D, two, count, sid, srow, n, cell_out, out, found);
}

// seeded lattice: ion g = site * per_site + p sits at its site plus a
// Gaussian jitter (normals D g + a of the jitter stream) and takes momenta
// sigma N (normals 3 g + a of the momentum stream); written as FP64 position
// and momentum rows for the load conversion
__device__ __forceinline__ double sm64_normal(uint64_t key, uint64_t c) {
  const double u1 = sm64_uniform(key, 2 * c), u2 = sm64_uniform(key, 2 * c + 1);
  return sqrt(-2.0 * log(1.0 - u1)) * cos(6.283185307179586476925 * u2);
}

__global__ void k_gen_lattice(int D, const double *sites, int per_site, double jitter, uint64_t kj, uint64_t km,
                              double sigma, const int *site_param, long long first, long long count, double *x,
                              double *u, int *pidx) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < count;
       q += (long long)gridDim.x * blockDim.x) {
    const long long gi = first + q, site = gi / per_site;
    for (int a = 0; a < D; ++a)
      x[q * D + a] = sites[site * D + a] + (jitter > 0.0 ? jitter * sm64_normal(kj, (uint64_t)(D * gi + a)) : 0.0);
    for (int a = 0; a < 3; ++a) u[q * 3 + a] = sigma > 0.0 ? sigma * sm64_normal(km, (uint64_t)(3 * gi + a)) : 0.0;
    if (pidx) pidx[q] = site_param[site];
  }
}

void launch_gen_lattice(int D, const double *sites, int per_site, double jitter, uint64_t seed, double sigma,
                        const int *site_param, long long first, long long count, double *x, double *u, int *pidx,
                        cudaStream_t s) {
  k_gen_lattice<<<blocks_for(count, 256), 256, 0, s>>>(D, sites, per_site, jitter, sm64_key(seed, 2),
                                                        sm64_key(seed, 3), sigma, site_param, first, count, x, u,
                                                        pidx);
}

void launch_gen_medium(const GridP &g, const SpecP &sp, PartP &p, const int lo[3], const int hi[3], int ppc,
                       uint64_t seed, double sigma, long long first, long long count, cudaStream_t s) {
  uint64_t kpos = sm64_key(seed, 1), kmom = sm64_key(seed, 3);
  k_gen_medium<<<blocks_for(count, 256), 256, 0, s>>>(g, sp, p, lo[0], lo[1], lo[2], hi[0] - lo[0], hi[1] - lo[1], ppc,
                                                       kpos, kmom, sigma, first, count, first);
}

void launch_rho(const GridP &g, const SpecP &sp, const PartP &p, double *rho, cudaStream_t s) {
  k_rho<<<blocks_for(p.cap, 256), 256, 0, s>>>(g, sp, p, rho);
}

void launch_divE_minus(const GridP &g, const float *const E[3], double *R, cudaStream_t s) {
  k_divE<<<blocks_for(g.ncell, 256), 256, 0, s>>>(g, E[0], E[1], E[2], R);
}

void launch_load_convert(const GridP &g, const SpecP &sp, PartP &p, const double *x, const double *u, const int *pidx,
                         long long first, long long count, int *status, cudaStream_t s) {
  k_load_convert<<<blocks_for(count, 256), 256, 0, s>>>(g, sp, p, x, u, pidx, first, count, status);
}
