// dsmc_team.cuh -- the FP32 layout's fused step with a CTA per cell, for
// handles with fewer cells than the GPU has warp slots.  Included by
// dsmc_ops.cuh.
#pragma once

namespace dsmc {

constexpr int TEAM_WARPS = 4;

// k_fused (see there) with the four warps of a CTA on one cell: the first
// collides, all of them sample and move a share.  With few cells a step takes
// as long as one cell's chain of phases, whichever SMs idle: 200 cells of 200
// particles, 20.0 us a step with a warp per cell, 11.8 us with a CTA per cell.
// Which form a handle takes is timed (step_bins).  Shared memory as k_fused's,
// the warps' tiles together one tile of TEAM_WARPS * wtile particles; a larger
// cell collides in global memory (owners: a hash table over the tile) and
// passes through in chunks.
template <int DIM, bool BATCH>
__global__ void __launch_bounds__(TEAM_WARPS * 32, 8) k_fused_team(
    const __grid_constant__ Params<float> pk, Cases<float> cases, int ncells, PBuf<float> in, PBuf<float> out,
    const int32_t* start, int32_t* cnt_in, int32_t* cnt_out,
    float* sgmax, double* acc, double* comp, Ovf ovi, Ovf ovo, int ovf_cap,
    int32_t* zero, uint32_t step_c, uint32_t step_m, int flags, int wtile, int ncell_blocks,
    double* tally_g, unsigned long long* stats, int32_t* errflag,
    float* stg, float* stc) {
  constexpr int NT = TEAM_WARPS * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned s_cnt[4];
  __shared__ unsigned s_misc[2];
  __shared__ float s_tally[20];
  __shared__ unsigned long long s_hits[2];
  __shared__ int s_nb[12];     // per destination: particles bound there
  __shared__ int2 s_slot[12];  // ... the first reserved slot in the arrays, slots that fit
  __shared__ float s_part[TEAM_WARPS][NMOM];
  __shared__ __align__(8) uint64_t s_bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < 4) s_cnt[tid] = 0;
  if (tid < 2) s_misc[tid] = 0;
  if (tid < 20) s_tally[tid] = 0.f;
  if (tid < 2) s_hits[tid] = 0;
  if (tid == 0) mbar_init(&s_bar, 1);
  mbar_fence_init();
  __syncthreads();
  grid_dep_wait();  // the previous launch filled the bins read here
  grid_dep_launch();
  if (blockIdx.x == 0 && tid == 0) *zero = 0;  // the next launch's output overflow counter
  if ((int)blockIdx.x < ncell_blocks) {
    const int tile = TEAM_WARPS * wtile;
    const int cell = blockIdx.x;
    const int cs = BATCH ? cases.cell_case[cell] : 0;
    const Params<float>& p = BATCH ? cases.p[cs] : pk;
    const int c0 = BATCH ? cases.cell0[cs] : 0;
    const int lcell = cell - c0;
    const int base = start[cell], n = cnt_in[cell];
    const bool fold = (flags & FF_FOLD) != 0;
    double pre[2] = {0.0, 0.0};
    float pre32[2] = {0.f, 0.f};
    const int mom = halving_moment(lane);
    if ((flags & FF_SAMPLE) && mom >= 0 && warp == 0) {
      pre32[0] = stg[(size_t)cell * NMOM + mom];
      pre32[1] = stc[(size_t)cell * NMOM + mom];
      if (fold) {
        pre[0] = acc[(size_t)cell * NMOM + mom];
        pre[1] = comp[(size_t)cell * NMOM + mom];
      }
    }
    float* vx = reinterpret_cast<float*>(smem);
    float* vy = vx + tile;
    float* vz = vx + 2 * tile;
    float* ir = vx + 3 * tile;
    const float* px = vx + 4 * tile;
    const float* py = vx + 5 * tile;
    uint32_t* own = reinterpret_cast<uint32_t*>(vx + 6 * tile);
    const bool staged = n <= tile;
    // bulk copies of particles [q0, q0 + m) of the cell into the tile at phase
    // ph of the barrier; bounded wait by every thread (false on a timeout)
    auto stage = [&](int q0, int m, uint32_t ph) -> bool {
      if (tid == 0) {
        constexpr int narr = (DIM == 2) ? 6 : 5;
        const uint32_t bytes = (uint32_t)((m + 3) & ~3) * 4u;
        const size_t o = (size_t)base + q0;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s_bar, bytes * narr);
        bulk_g2s(vx, in.vx + o, bytes, &s_bar);
        bulk_g2s(vx + tile, in.vy + o, bytes, &s_bar);
        bulk_g2s(vx + 2 * tile, in.vz + o, bytes, &s_bar);
        bulk_g2s(vx + 3 * tile, in.ir + o, bytes, &s_bar);
        bulk_g2s(vx + 4 * tile, in.x + o, bytes, &s_bar);
        if (DIM == 2) bulk_g2s(vx + 5 * tile, in.y + o, bytes, &s_bar);
      }
      const bool r = mbar_wait_bounded(&s_bar, ph, MBAR_POLL_LIMIT);
      if (!r) atomicOr(errflag, 1);
      return __syncthreads_and(r) != 0;
    };
    bool ok = true;
    if (staged && n > 0) ok = stage(0, n, 0u);
    if ((flags & FF_COLLIDE) && ok) {
      if (warp == 0) {
        const float sgm = sgmax[cell];
        const uint32_t M = ntc_candidates<float>(p, n, (uint32_t)lcell, step_c, sgm);
        CollCount cc{0, 0, 0, 0};
        if (M != 0u && staged)
          collide_window<float, false, 32>(p, vx, vy, vz, ir, n, (uint32_t)lcell, step_c, sgm, M, sgmax + cell, own,
                                           cc);
        else if (M != 0u)
          collide_window<float, false, 32>(p, in.vx + base, in.vy + base, in.vz + base, in.ir + base, n,
                                           (uint32_t)lcell, step_c, sgm, M, sgmax + cell,
                                           reinterpret_cast<uint32_t*>(vx), cc,
                                           (0x80000000u >> __clz(7 * tile)) - 1u);
        flush_counts<float>(cc, s_cnt);
        if (!staged) fence_proxy_async_global();  // the bulk copies below read these velocities
      }
      __syncthreads();
    }
    float mtot = 0.f;  // this lane's moment over the warp's shares
    const int cix = lcell % p.nx, ciy = lcell / p.nx;
    uint32_t ph = 0u;
    for (int q0 = 0; q0 < n && ok; q0 += tile) {
      const int m = min(tile, n - q0);
      if (!staged) {
        __syncthreads();  // every thread is done with the previous chunk
        ok = stage(q0, m, ph);
        ph ^= 1u;
        if (!ok) break;
      }
      if (tid < 12) s_nb[tid] = 0;
      if (flags & FF_SAMPLE) {
        const int share = ((m + NT - 1) / NT) * 32;
        const int a = min(m, warp * share), b = min(m, a + share);
        mtot += sample_chunk(vx + a, vy + a, vz + a, ir + a, b - a);
      }
      __syncthreads();
      // M1: destinations and ranks
      for (int q = tid; q < m; q += NT) {
        float xn, yn;
        int code = 9;
        if (flight_stays_inside<float, DIM>(p, px[q], (DIM == 2) ? py[q] : 0.f, vx[q], vy[q], &xn, &yn))
          code = neighbour_code<DIM>(p, cix, ciy, xn, yn);
        const int r = atomicAdd(&s_nb[code], 1);
        own[q] = ((uint32_t)code << 24) | (uint32_t)r;
      }
      __syncthreads();
      // M2: reserve the slots, one atomic per destination bin
      if (tid < 9 && s_nb[tid] > 0) {
        const int want = s_nb[tid], d = neighbour_cell(p.nx, cell, tid);
        const int b0 = atomicAdd(&cnt_out[d], want);
        const int s0 = start[d], cap = start[d + 1] - s0;
        s_slot[tid] = make_int2(s0 + b0, cap - b0);
        if (b0 + want > cap - 8) atomicAdd(s_misc + 1, 1u);
      }
      __syncthreads();
      // M3: store; a particle that reaches a wall or goes far is flown in
      // full, with wall tallies
      for (int q = tid; q < m; q += NT) {
        float x = px[q], y = (DIM == 2) ? py[q] : 0.f;
        float a = vx[q], b = vy[q], c = vz[q], e = ir[q];
        const uint32_t tag = own[q];
        const int code = (int)(tag >> 24), r = (int)(tag & 0xFFFFFFu);
        int d = -1, w;
        bool fits;
        if (code < 9) {
          x = x + a * p.dt;
          if (DIM == 2) y = y + b * p.dt;
          const int2 sl = s_slot[code];
          w = sl.x + r;
          fits = r < sl.y;
        } else {
          fly<float, DIM, true, false>(p, x, y, a, b, c, e, (uint32_t)(q0 + q), (uint32_t)lcell, step_m, s_tally,
                                       &s_hits[0], &s_hits[1]);
          d = c0 + cell_of<float, DIM>(p, x, y);
          const int slot = atomicAdd(&cnt_out[d], 1);
          const int s0 = start[d], cap = start[d + 1] - s0;
          w = s0 + slot;
          fits = slot < cap;
          if (slot >= cap - 8) atomicAdd(s_misc + 1, 1u);
        }
        if (fits) {
          out.x[w] = x;
          if (DIM == 2) out.y[w] = y;
          out.vx[w] = a;
          out.vy[w] = b;
          out.vz[w] = c;
          out.ir[w] = e;
        } else {
          // reserved but unused slot: give it back (the bin's count ends at
          // its capacity)
          if (d < 0) d = neighbour_cell(p.nx, cell, code);
          atomicSub(&cnt_out[d], 1);
          const int qo = atomicAdd(ovo.count, 1);
          atomicAdd(s_misc + 0, 1u);
          if (qo < ovf_cap) {
            ovo.x[qo] = x;
            ovo.y[qo] = y;
            ovo.vx[qo] = a;
            ovo.vy[qo] = b;
            ovo.vz[qo] = c;
            ovo.ir[qo] = e;
            ovo.dest[qo] = d;
          } else {
            atomicOr(errflag, 2);  // the overflow list is full: the particle is lost
          }
        }
      }
    }
    if (ok) {
      if (flags & FF_SAMPLE) {
        if (mom >= 0) s_part[warp][mom] = mtot;
        __syncthreads();
        if (warp == 0) {
          if (mom >= 0) {
            mtot = s_part[0][mom];
#pragma unroll
            for (int v = 1; v < TEAM_WARPS; ++v) mtot += s_part[v][mom];
          }
          sample_fold(mtot, mom, acc + (size_t)cell * NMOM, comp + (size_t)cell * NMOM, pre,
                      stg + (size_t)cell * NMOM, stc + (size_t)cell * NMOM, pre32, fold);
        }
      }
      if (tid == 0) cnt_in[cell] = 0;
    }
  } else {
    // overflow list of the previous step: move and append (no collision)
    const int nov = min(*ovi.count, ovf_cap);
    const int gw = (blockIdx.x - ncell_blocks) * TEAM_WARPS + warp;
    const int nwarps = (gridDim.x - ncell_blocks) * TEAM_WARPS;
    for (int base = gw * 32; base < nov; base += nwarps * 32) {
      const int q = base + lane;
      const bool active = q < nov;
      float x = 0.f, y = 0.f, a = 0.f, bb = 0.f, c = 0.f, e = 0.f;
      int d = 0;
      if (active) {
        const int cs = BATCH ? cases.cell_case[ovi.dest[q]] : 0;
        const Params<float>& p = BATCH ? cases.p[cs] : pk;
        const int c0 = BATCH ? cases.cell0[cs] : 0;
        x = ovi.x[q];
        y = ovi.y[q];
        a = ovi.vx[q];
        bb = ovi.vy[q];
        c = ovi.vz[q];
        e = ovi.ir[q];
        fly<float, DIM, true, false>(p, x, y, a, bb, c, e, (uint32_t)q, (uint32_t)(p.ncells + 1), step_m, s_tally,
                                     &s_hits[0], &s_hits[1]);
        d = c0 + cell_of<float, DIM>(p, x, y);
      }
      append_particle<DIM>(pk, out, start, cnt_out, ovo, ovf_cap, active, d, x, y, a, bb, c, e, s_misc, errflag);
    }
  }
  __syncthreads();
  if (tid < 4 && s_cnt[tid]) atomicAdd(stats + tid, (unsigned long long)s_cnt[tid]);
  if (tid == 4 && s_misc[0]) atomicAdd(stats + ST_OVF, (unsigned long long)s_misc[0]);
  if (tid == 5 && s_misc[1]) atomicAdd(stats + ST_NEARFULL, (unsigned long long)s_misc[1]);
  if (tid == 6 && s_hits[0]) atomicAdd(stats + ST_HITS, s_hits[0]);
  if (tid == 7 && s_hits[1]) atomicAdd(stats + ST_MAXHIT, s_hits[1]);
  if (tid < 20 && s_tally[tid] != 0.f) atomicAdd(tally_g + tid, (double)s_tally[tid]);
}

}  // namespace dsmc
