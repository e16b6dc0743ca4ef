// The FP64 step's sweep.  GB300 issues an FP64 instruction per SM only every
// ~19 cycles, whatever the number of active lanes, so the FP64 form is bound
// by how many lanes of a warp work: with one thread per column, warps of 32
// unrelated columns ran the processes with 13.4 lanes on average (stratus,
// 30 % cloudy columns), and the long inlined code of the branches they took
// one after the other missed the instruction cache.
//
// Here a block of 128 threads takes 32 columns and walks them down in chunks of levels.  In
// each chunk it flags the points (every lane busy), lists the active ones by
// the branches they will take, runs the processes over the list in full
// warps, and then applies the sedimentation, whose fluxes the points hand
// down through shared memory: a level's outgoing flux depends on its own
// point alone, so only the update needs the level above.
// Measured: FP64 step, 256x256x100 stratus 28.7 -> 9.9 ms (24.7 lanes, FP64
// pipe 66 % busy over the launch instead of 45 %), deep convection of that size
// 35.5 -> 16.9 ms, 2 000 columns 5.2 -> 0.52 ms; with exp, log and the quotients
// out of line or cheaper (casim_math64.cuh, the same bits), flags decided in FP32
// away from saturation and comparisons on the integer pipe (an FP64 compare
// costs as much as an addition) 6.0, 10.6 and 0.37 ms.
// (included by casim_device.cuh)
#pragma once

namespace casim_dev {

constexpr int kF64Cols = 32;      // columns of a tile
// levels of a chunk.  At 32 levels of 8 fluxes a point the tile is 76 KB, two
// blocks to an SM; at 16 levels of 12 fluxes (sixth moments, aerosol mass) three.
// Measured, cold step, 24 levels (three blocks) / 32 levels: 65 536 x 100
// stratus 5.84 / 5.96 ms, deep convection 10.97 / 10.47; 16 384 x 150 deep
// convection 6.5 / 4.9 (an item of 150 levels is 7 chunks, or 5)
template <class M>
__host__ __device__ constexpr int f64_levels() {
  return M::kWarm || M::kTri || M::kAero ? 16 : 32;
}
template <class M>
__host__ __device__ constexpr int f64_points() {   // row 0: the level above the chunk
  return (f64_levels<M>() + 1) * kF64Cols;
}
constexpr int kF64Classes = 3;

// x != 0 on the integer pipe
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) & 0x7fffffffffffffffll) != 0; }

// flux arrays: mass and number of each sedimenting species, and its sixth
// moment or aerosol mass
template <class M>
__host__ __device__ constexpr int f64_fluxes() {
  return (M::kWarm ? 1 : 4) * (M::kTri || M::kAero ? 3 : 2);
}

template <class M>
struct F64Tile {
  static constexpr int kPts = f64_points<M>();
  double flux[f64_fluxes<M>()][kPts];
  double halo[22][kF64Cols];                    // the level above the segment, as read
  unsigned long long cmax[4][kF64Cols];         // multi-substep path: largest Courant numbers (bits)
  int cnt[kF64Classes + 1];
  int col[kF64Cols];                            // the tile's columns, -1: none
  unsigned short list[kPts];                 // active points, by class
  unsigned char cls[kPts];                   // 0: inactive, else 1 + class
};

// Statistics of a tile's columns (the statistics instantiation).
struct F64Stats {
  int active[kF64Cols], nsub[4][kF64Cols];
  unsigned lv[kF64Cols][(kMaxLev + 31) / 32];   // levels the step changed
};

// One tile: 32 columns (t.col), the levels of sg.  Every thread of the block
// calls it.  Results are those of the process chain and sedimentation point
// by point, in the order of the levels, as sweep_column's.
// st: the statistics instantiation's counters, or null.
template <class M, bool kTend, bool kStats = false>
__device__ __forceinline__ unsigned f64_sweep(const KArgs &a, const KParams &P, const LevelTab &lt, bool fast,
                                              const Segment<true> &sg, double *tend, F64Tile<M> &t,
                                              F64Stats *st = nullptr) {
  static_assert(!M::kMixed, "FP64 policies");
  using Ph = Phys<M>;
  const ConstK<double> &K = P.d;
  constexpr int kSed = M::kWarm ? 1 : 4;
  constexpr int kF = M::kTri || M::kAero ? 3 : 2;   // fluxes per species
  const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const size_t fs = (size_t)a.nlev * (size_t)a.pitch;
  const DtDiv per_dt(kTend ? a.dt : 1.0);
  const bool halo = fast && sg.seg > 0, share = !kTend && fast && sg.nseg > 1;
  unsigned eflag = 0;
  for (int i = tid; i < 4 * kF64Cols; i += B) t.cmax[i / kF64Cols][i % kF64Cols] = 0ull;
  for (int i = tid; i < f64_fluxes<M>() * kF64Cols; i += B) t.flux[i / kF64Cols][i % kF64Cols] = 0.0;
  if constexpr (kStats) {
    for (int i = tid; i < kF64Cols; i += B) {
      st->active[i] = 0;
      for (int x = 0; x < 4; ++x) st->nsub[x][i] = 1;
      for (unsigned &w : st->lv[i]) w = 0u;
    }
  }
  for (int ktop = sg.ktop(); ktop >= sg.kbot(); ktop -= f64_levels<M>()) {
    const bool first = ktop == sg.ktop();
    const int rows = 1 + min(f64_levels<M>(), ktop - sg.kbot() + 1);
    const int i0 = first && halo ? 0 : kF64Cols, i1 = rows * kF64Cols;   // this chunk's points
    if (tid <= kF64Classes) t.cnt[tid] = 0;
    __syncthreads();
    // 1. flag the points
    for (int i = i0 + tid; i < i1; i += B) {
      const int row = i >> 5, k = ktop + 1 - row, c = t.col[lane];
      unsigned cls = 0;
      if (c >= 0) {
        Pt s;
        load_pt<M::kWarm, M::kAero, M::kTri>(a, k, c, s);
        eflag |= nonfinite_in(s);
#pragma unroll
        for (int e = 0; e < nextra<M>(); ++e) eflag |= nonfinite(extra<M>(s, e));
        if (row == 0) {
#pragma unroll
          for (int f = 0; f < 16 + nextra<M>(); ++f) t.halo[f][lane] = pt_field<M>(s, f);
        }
        cls = F64T<M>::flag(K, P.f, s);
      }
      t.cls[i] = (unsigned char)cls;
      if constexpr (kStats) {
        if (cls) {
          atomicAdd(&st->active[lane], 1);
          atomicOr(&st->lv[lane][k >> 5], 1u << (k & 31));
        }
      }
#pragma unroll
      for (int f = 0; f < f64_fluxes<M>(); ++f) t.flux[f][i] = 0.0;
#pragma unroll
      for (int j = 1; j <= kF64Classes; ++j) {
        const unsigned b = __ballot_sync(0xffffffffu, cls == j);
        if (lane == 0 && b) atomicAdd(&t.cnt[j], __popc(b));
      }
    }
    if (share && first) split_arrive();   // the level above the segment has been read
    __syncthreads();
    const int n1 = t.cnt[1], n2 = t.cnt[2], total = n1 + n2 + t.cnt[3];
    __syncthreads();
    // 2. list the active ones by class
    if (tid <= kF64Classes) t.cnt[tid] = tid == 1 ? 0 : tid == 2 ? n1 : n1 + n2;
    __syncthreads();
    for (int i = i0 + tid; i < i1; i += B) {
      const unsigned cls = t.cls[i];
#pragma unroll
      for (int j = 1; j <= kF64Classes; ++j) {
        const unsigned b = __ballot_sync(0xffffffffu, cls == j);
        int at = 0;
        if (lane == 0 && b) at = atomicAdd(&t.cnt[j], __popc(b));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (cls == j) t.list[at + __popc(b & ((1u << lane) - 1u))] = (unsigned short)i;
      }
    }
    if (share && first) split_wait();
    __syncthreads();
    // 3. the processes and outgoing fluxes of the listed points
    for (int base = warp * 32; base < total; base += B) {
      if (base + lane < total) {
        const int i = t.list[base + lane], row = i >> 5, col = i & 31, k = ktop + 1 - row, c = t.col[col];
        Pt s;
        if (row == 0) {
          if constexpr (M::kWarm) s.qi = s.qs = s.qg = s.ni = s.ns = s.ng = 0.0;
#pragma unroll
          for (int f = 0; f < 16 + nextra<M>(); ++f) {
            const bool ice = (f >= 4 && f <= 6) || (f >= 9 && f <= 11);
            if (!(M::kWarm && ice)) pt_field<M>(s, f) = t.halo[f][col];
          }
        } else {
          load_pt<M::kWarm, M::kAero, M::kTri>(a, k, c, s);
        }
        double mu3[4];
        unsigned keep3 = 0;   // species whose shape the processes left unchanged (triple-moment policies)
        double dfac;
        F64T<M>::process(K, s, a.dt, t.cls[i] < 3, dfac, mu3, &keep3);
        if (fast) {
          bool any = false;
#pragma unroll
          for (int x = 0; x < kSed; ++x) any |= M::gt(qref(s, x), K.qmin);
          if (any) {
            if (dfac == 0.0) dfac = exp64(0.4 * (K.lgrho0 - log64(s.rho)));
#pragma unroll
            for (int x = 0; x < kSed; ++x) {
              const double q = qref(s, x), n = nref(s, x);
              if (!M::gt(q, K.qmin)) continue;
              double vq, vn;
              if (x < nz3<M>()) {
                double vz;
                const double z = zref(s, x);
                const double mus = ((keep3 >> x) & 1u) ? mu3[x] : Shape3<M>::mu(K, x, q, n, z);
                Shape3<M>::fall_speeds_mu(K, x, lt.dzdt[k], log64(q), n, mus, dfac, vq, vn, vz);
                t.flux[kF * x + 2][i] = s.rho * (z > 0.0 ? z : 0.0) * vz;
              } else {
                Ph::fall_speeds(K, lt.dzdt[k], q, n, dfac, x, vq, vn);
              }
              t.flux[kF * x][i] = s.rho * q * vq;
              t.flux[kF * x + 1][i] = s.rho * M::pos(n) * vn;
              if (x < na3<M>()) t.flux[kF * x + 2][i] = s.rho * maref(s, x) * vq;
            }
          }
        } else {
          double cm[4] = {0.0, 0.0, 0.0, 0.0};
          courant<M>(a, K, lt.dz, k, s, cm);
#pragma unroll
          for (int x = 0; x < kSed; ++x)
            if (cm[x] > 0.0) atomicMax(&t.cmax[x][col], (unsigned long long)__double_as_longlong(cm[x]));
        }
        if (row > 0) {
          if constexpr (kTend) {
            eflag |= store_tend<M>(a, tend, k, c, s, false, per_dt);   // the new values; source terms below
          } else if constexpr (M::kWarm) {
            eflag |= store_pt_warm<M::kAero, M::kTri>(a, k, c, s);
          } else {
            eflag |= store_pt(a, k, c, s);
            double *b = a.fld + (size_t)k * a.pitch + c;
#pragma unroll
            for (int e = 0; e < nextra<M>(); ++e) {
              b[(16 + e) * fs] = extra<M>(s, e);
              eflag |= nonfinite(extra<M>(s, e));
            }
          }
        }
      }
    }
    __syncthreads();
    // 4. sedimentation (single-substep path) and source terms
    if (fast || kTend) {
      for (int i = kF64Cols + tid; i < i1; i += B) {
        const int k = ktop + 1 - (i >> 5), c = t.col[lane];
        if (c < 0) continue;
        const size_t o = (size_t)k * a.pitch + c;
        const bool act = t.cls[i] != 0;
        double *out = kTend ? tend : a.fld;
        const double *in = kTend && act ? tend : a.fld;   // where the processed values are
        Div64 per_mass;      // divides by rho dz
        bool have = false;   // some species moves here
#pragma unroll
        for (int x = 0; x < kSed; ++x) {
          const double F = t.flux[kF * x][i], F1 = t.flux[kF * x][i - kF64Cols];
          const double G = t.flux[kF * x + 1][i], G1 = t.flux[kF * x + 1][i - kF64Cols];
          const bool wq = fast && (nonzero(F) || nonzero(F1) || nonzero(G) || nonzero(G1));
          double X = 0.0, X1 = 0.0;
          if constexpr (kF == 3) {
            X = t.flux[kF * x + 2][i];
            X1 = t.flux[kF * x + 2][i - kF64Cols];
          }
          const bool wx = fast && (nonzero(X) || nonzero(X1));
          if ((wq || wx) && !have) {
            per_mass = Div64(__ldg(a.fld + 14 * fs + o) * lt.dz[k]);
            have = true;
          }
          // field 16 + x: a sixth moment; 18 + x: an aerosol mass (source-term row: three less)
          const int fx = M::kTri ? 16 + x : 18 + x, rx = kTend ? fx - 3 : fx, ix = kTend && act ? fx - 3 : fx;
          if (wq || kTend) {
            double q = in[(3 + x) * fs + o], n = in[(8 + x) * fs + o];
            if (wq) {
              q += per_mass(a.dt * (F1 - F));
              n += per_mass(a.dt * (G1 - G));
              eflag |= nonfinite(q) | nonfinite(n);
            }
            if (kTend && fast) {
              q = per_dt(q - a.fld[(3 + x) * fs + o]);
              n = per_dt(n - a.fld[(8 + x) * fs + o]);
            }
            out[(3 + x) * fs + o] = q;
            out[(8 + x) * fs + o] = n;
          }
          if constexpr (kF == 3) {
            if (wx || kTend) {
              double e = in[ix * fs + o];
              if (wx) {
                e += per_mass(a.dt * (X1 - X));
                eflag |= nonfinite(e);
              }
              if (kTend && fast) e = per_dt(e - a.fld[fx * fs + o]);
              out[rx * fs + o] = e;
            }
          }
        }
        if constexpr (kStats) {
          if (have) atomicOr(&st->lv[lane][k >> 5], 1u << (k & 31));
        }
        if constexpr (kTend) {
          // the fields that do not sediment (multi-substep path: the new
          // values, which the sweeps read; source terms afterwards)
#pragma unroll
          for (int f = 0; f < 13; ++f) {
            const bool ice = (f >= 4 && f <= 6) || (f >= 9 && f <= 11);
            const bool sed = M::kWarm ? f == 3 || f == 8 : (f >= 3 && f <= 6) || (f >= 8 && f <= 11);
            if (sed) continue;
            if (M::kWarm && ice) tend[f * fs + o] = 0.0;
            else if (fast) tend[f * fs + o] = per_dt(in[f * fs + o] - a.fld[f * fs + o]);
            else if (!act) tend[f * fs + o] = a.fld[f * fs + o];
          }
#pragma unroll
          for (int e = 0; e < nextra<M>(); ++e) {
            if (M::kTri || e >= 2 && e < 2 + kSed) continue;   // the species' own: above
            const double v = act ? tend[(13 + e) * fs + o] : a.fld[(16 + e) * fs + o];
            tend[(13 + e) * fs + o] = fast ? per_dt(v - a.fld[(16 + e) * fs + o]) : v;
          }
        }
      }
      __syncthreads();
      // the fluxes out of the chunk, for the one below
      for (int i = tid; i < f64_fluxes<M>() * kF64Cols; i += B)
        t.flux[i / kF64Cols][i % kF64Cols] = t.flux[i / kF64Cols][i1 - kF64Cols + i % kF64Cols];
    }
  }
  __syncthreads();
  double prec[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (fast) {
    if (sg.kbot() == 0 && warp == 0) {
#pragma unroll
      for (int x = 0; x < kSed; ++x) {
        prec[x] = t.flux[kF * x][lane] * a.dt;
        if constexpr (M::kAero) prec[4] += t.flux[kF * x + 2][lane] * a.dt;
      }
    }
  } else {
    // the segments' Courant numbers meet in the top segment's block, whose warps
    // take a species each (with aerosol mass one thread takes them all: their
    // surface fluxes of aerosol add up in order).  The other blocks leave, so that
    // a cluster of a later wave need not wait for the sweeps (1 824 columns x 60,
    // dt = 10 s, 8 segments: 2.80 -> 1.68 ms, source terms 2.83 -> 1.80).
    auto barrier = [&] {
      if (sg.nseg > 1) {
        split_arrive();
        split_wait();
      }
    };
    barrier();
    const int c = t.col[lane];
    double cmax[4] = {0.0, 0.0, 0.0, 0.0};
    if (sg.seg == 0) {
#pragma unroll
      for (int x = 0; x < kSed; ++x) {
        for (int j = 0; j < sg.nseg; ++j) {
          const double v = sg.nseg > 1 ? sg.slot(reinterpret_cast<const double *>(&t.cmax[x][lane]), j)
                                       : __longlong_as_double((long long)t.cmax[x][lane]);
          cmax[x] = v > cmax[x] ? v : cmax[x];
        }
      }
    }
    barrier();   // the slots have been read
    constexpr int kPass = kStats ? 32 : pass_substeps<M, false>();   // (the statistics hold local memory too)
    for (int x = 0; x < kSed; ++x) {
      const bool mine = sg.seg == 0 && warp == (M::kAero ? 0 : x % (B >> 5));
      if (!mine || c < 0) continue;
      int ns = (int)ceil((x == 0 ? cmax[0] : x == 1 ? cmax[1] : x == 2 ? cmax[2] : cmax[3]) / P.c_max);
      if (ns < 1) ns = 1;
      if (ns > 64) { ns = 64; eflag |= 2u; }
      double pr = 0.0;
      if constexpr (kStats) {
        unsigned lv[(kMaxLev + 31) / 32] = {};
        st->nsub[x][lane] = ns;
        eflag |= sediment_species<M, kTend, kPass>(a, P, lt, c, x, ns, pr, prec[4], tend, lv);
        for (int w = 0; w < (kMaxLev + 31) / 32; ++w)
          if (lv[w]) atomicOr(&st->lv[lane][w], lv[w]);
      } else {
        eflag |= sediment_species<M, kTend, kPass>(a, P, lt, c, x, ns, pr, prec[4], tend, nullptr);
      }
#pragma unroll
      for (int j = 0; j < kSed; ++j)
        if (x == j) prec[j] = pr;
    }
    __syncthreads();
    if constexpr (kTend) {
      for (int i = tid; i < (sg.seg == 0 ? a.nlev * kF64Cols : 0); i += B) {
        const int k = i >> 5;
        if (c < 0) continue;
        const size_t o = (size_t)k * a.pitch + c;
#pragma unroll
        for (int f = 0; f < 13; ++f) {
          const bool ice = (f >= 4 && f <= 6) || (f >= 9 && f <= 11);
          if (!(M::kWarm && ice)) tend[f * fs + o] = per_dt(tend[f * fs + o] - a.fld[f * fs + o]);
        }
#pragma unroll
        for (int e = 0; e < nextra<M>(); ++e)
          tend[(13 + e) * fs + o] = per_dt(tend[(13 + e) * fs + o] - a.fld[(16 + e) * fs + o]);
      }
    }
  }
  const int c = t.col[lane];
  if (c >= 0) {
#pragma unroll
    for (int x = 0; x < 5; ++x) {
      if (x >= kSed && !(M::kAero && x == 4)) continue;
      if (prec[x] != 0.0 && CASIM_INDEX_OK(c < a.ncols, a.err)) {
        double *pp = a.precip + (size_t)x * a.pitch + c;
        *pp += prec[x];
        eflag |= nonfinite(*pp);
      }
    }
  }
  __syncthreads();   // the tile's shared memory is free again
  if constexpr (kStats) {
    if (warp == 0 && c >= 0) {
      ColStats cs{st->active[lane], 0, {st->nsub[0][lane], st->nsub[1][lane], st->nsub[2][lane], st->nsub[3][lane]}};
      for (unsigned w : st->lv[lane]) cs.changed += __popc(w);
      stats_add(a.stats, cs);
    }
  }
  return eflag;
}

}  // namespace casim_dev
