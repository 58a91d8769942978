// Host check of the ordered recursion (ordered.h): for every process given on
// the command line and a few phase-space points of the input generator, the
// helicity- and colour-summed |M|^2 must equal the per-lane program's (every
// Feynman diagram and helicity combination, the program's colour basis).
// Stages run level by level; nothing may be read that the level writes or that
// was never written, and every access lies inside its array.  Prints per
// process: name, largest relative difference, doubles and amplitudes per event;
// exit status 1 on a fault.
#define MEA_HD inline
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../paper_0909_5257_gb300/phasespace/phasespace.h"
#include "ordered_eval.cuh"

using namespace mea;

static int faults = 0;

int main(int argc, char** argv) {
  for (int arg = 1; arg < argc; ++arg) {
    std::vector<int> pdg;
    std::string s = argv[arg];
    for (size_t p = 0; p < s.size();) {
      size_t e = s.find(',', p);
      if (e == std::string::npos) e = s.size();
      pdg.push_back(std::atoi(s.substr(p, e - p).c_str()));
      p = e + 1;
    }
    const Program P = build_program(pdg);
    const OrdProgram Q = build_ordered(P);
    const int n = P.n_ext, m = P.n_jamp;
    const double g = 1.2;
    std::vector<int8_t> leg(4 * n, 0);
    for (int l = 0; l < n; ++l) {
      leg[4 * l] = (int8_t)P.leg_type[l];
      leg[4 * l + 1] = (int8_t)(P.leg_type[l] == 1 ? (P.incoming[l] ? 0 : 1) : P.leg_type[l] == 2 ? (P.incoming[l] ? 3 : 2) : 0);
      leg[4 * l + 2] = (int8_t)P.incoming[l];
    }
    double worst = 0.0;
    for (int ev = 0; ev < (n == 7 ? 1 : 3); ++ev) {
      double mom[PS_MAX_FINAL + 2][4];
      ps_config cfg;
      std::memset(&cfg, 0, sizeof cfg);
      cfg.seed = 0x5eed;
      cfg.n_final = n - 2;
      cfg.rs_lo = 200;
      cfg.rs_hi = 2000;
      cfg.pt_min = 20;
      cfg.eta_max = 2.5;
      cfg.dr_min = 0.4;
      ps_generate_event(&cfg, (uint64_t)ev, mom);
      // event table (amp_common.cuh)
      std::vector<double> et(8 * n, 0.0), mt(5 * P.masks.size(), 0.0);
      for (int l = 0; l < n; ++l) {
        const double *p = mom[l], px = p[1], py = p[2], pz = p[3];
        double* o = &et[8 * l];
        const double kt2 = px * px + py * py, kk = std::sqrt(kt2 + pz * pz), kt = std::sqrt(kt2);
        if (P.leg_type[l] == 0) {
          const double ct = kt > 0 ? pz / kk : (pz < 0 ? -1 : 1), st = kt > 0 ? kt / kk : 0, cp = kt > 0 ? px / kt : 1, sp = kt > 0 ? py / kt : 0;
          o[0] = ct * cp; o[1] = ct * sp; o[2] = -st; o[3] = -sp; o[4] = cp; o[5] = 0;
        } else {
          const double apz = pz >= 0 ? kk + pz : kt2 / (kk - pz);
          o[0] = std::sqrt(2 * p[0]);
          if (apz > 0) {
            const double nrm = 1 / std::sqrt(2 * kk * apz);
            o[1] = apz * nrm; o[2] = px * nrm; o[3] = py * nrm;
          } else {
            o[1] = 0; o[2] = 1; o[3] = 0;
          }
        }
      }
      for (size_t r = 0; r < P.masks.size(); ++r) {
        double* q = &mt[5 * r];
        for (int l = 0; l < n; ++l)
          if (P.masks[r] >> l & 1u)
            for (int k = 0; k < 4; ++k) q[k] += (P.incoming[l] ? -1.0 : 1.0) * mom[l][k];
        if (__builtin_popcount(P.masks[r]) > 1) q[4] = 1 / (q[0] * q[0] - q[1] * q[1] - q[2] * q[2] - q[3] * q[3]);
      }
      // every diagram of every combination
      long double ref = 0.0;
      for (int h = 0; h < P.n_hel; ++h) {
        std::vector<W4<double>> slots(P.n_slots);
        std::vector<cx<double>> J(m, cx<double>{0, 0});
        const double* M = mt.data();
        for (const Op& op : P.ops) {
          W4<double> x[4];
          const int n_in = op.type == OP_EXT ? 0 : op.n_in;
          for (int k = 0; k < n_in; ++k) x[k] = slots[op.in[k]];
          cx<double> a{0, 0};
          W4<double> w{};
          const double *k0 = M + 5 * op.min[0], *k1 = M + 5 * op.min[1], *k2 = M + 5 * op.min[2], *q = M + 5 * op.mout;
          switch (op.type) {
            case OP_EXT: {
              const double* o = &et[8 * op.leg];
              const int lam = P.hel[(size_t)h * n + op.leg];
              w = P.leg_type[op.leg] == 0 ? ext_gluon<double>(o, o + 3, lam, !P.incoming[op.leg])
                                          : ext_spinor<double>(o[0], o[1], mk<double>(o[2], o[3]), lam, leg[4 * op.leg + 1]);
              break;
            }
            case OP_JVV: w = jvv<double>(x[0], x[1], k0, k1, q[4], g); break;
            case OP_JGGG: w = jggg<double>(x[0], x[1], x[2], q[4], g * g); break;
            case OP_FVI: w = fvi<double>(x[0], x[1], q, q[4], g); break;
            case OP_FVO: w = fvo<double>(x[0], x[1], q, q[4], g); break;
            case OP_JIO: w = jio<double>(x[0], x[1], q[4], g); break;
            case OP_PVVV: w = vvv_part<double>(x[0], x[1], k0, k1, k2, g); break;
            case OP_PGGGG: w = gggg_part<double>(x[0], x[1], x[2], g * g); break;
            case OP_PIOV: w = op.leg == 0 ? iov_part_i<double>(x[0], x[1], g) : op.leg == 1 ? iov_part_o<double>(x[0], x[1], g) : iov_part_v<double>(x[0], x[1], g); break;
            case OP_AVVV: a = vvv_amp<double>(x[0], x[1], x[2], k0, k1, k2, g); break;
            case OP_AGGGG: a = gggg_amp<double>(x[0], x[1], x[2], x[3], g * g); break;
            case OP_AIOV: a = iov_amp<double>(x[0], x[1], x[2], g); break;
            case OP_ADOT: a = part_contract<double>(x[0], x[1], op.leg & 1, op.leg & 2); break;
          }
          if (!is_amp_op(op.type)) { slots[op.out] = w; continue; }
          for (uint32_t k = 0; k < op.col_count; ++k) {
            const ColEntry& c = P.col[op.col_begin + k];
            J[c.alpha] = J[c.alpha] + mk<double>(c.re, c.im) * a;
          }
        }
        for (int a = 0; a < m; ++a)
          for (int b = 0; b < m; ++b) ref += (long double)P.cf_jamp[(size_t)a * m + b] * (J[a].r * J[b].r + J[a].i * J[b].i) / (double)P.cf_den;
      }
      // ordered recursion; NaN marks what is not written
      const double nan = std::nan("");
      std::vector<double> area(Q.area, nan), F(2 * Q.n_f, nan);
      for (size_t i = 0; i < Q.stages.size();) {
        size_t j = i;
        while (j < Q.stages.size() && Q.level[j] == Q.level[i]) ++j;
        std::vector<double> next = area;  // a level reads what earlier levels wrote
        for (size_t q = i; q < j; ++q) {
          const OrdStage& st = Q.stages[q];
          for (int w = 0; w < st.words; ++w)
            for (uint32_t v = 0; v < (1u << st.nb); ++v) {
              std::vector<double> out = area;
              OrdEvent E{out.data(), F.data(), et.data(), mt.data(), leg.data()};
              if (n >= 6) {  // the copies are for the small processes
                E.area = next.data();
                ord_item(st, Q.rec.data() + st.rec + (size_t)w * st.stride, v, E);
                continue;
              }
              ord_item(st, Q.rec.data() + st.rec + (size_t)w * st.stride, v, E);
              for (size_t k = 0; k < out.size(); ++k)
                if (std::memcmp(&out[k], &area[k], 8)) {
                  if (next[k] == next[k]) ++faults, std::printf("written twice\n");
                  next[k] = out[k];
                }
            }
        }
        area = next;
        i = j;
      }
      long double got = 0.0;
      for (int h = 0; h < Q.H; ++h)
        for (int a = Q.range[2 * h]; a < Q.range[2 * h + 1]; ++a)
          for (int b = Q.range[2 * h]; b < Q.range[2 * h + 1]; ++b) {
            const double *x = &F[2 * Q.fidx[(size_t)a * Q.H + h]], *y = &F[2 * Q.fidx[(size_t)b * Q.H + h]];
            got += (long double)Q.kmat[(size_t)a * Q.n_colour + b] * (x[0] * y[0] + x[1] * y[1]);
          }
      got *= Q.norm * std::pow(g, 2 * n - 4);
      const double d = (double)std::fabs(got / ref - 1);
      if (!(d < 1e-11)) ++faults;
      worst = d < worst ? worst : d;
    }
    std::printf("%s %.2e %d %d\n", argv[arg], worst, Q.area, Q.n_f);
  }
  return faults ? 1 : 0;
}
