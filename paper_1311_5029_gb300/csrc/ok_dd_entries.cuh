// The matrix-vector products of one application of M (Eq. minFlopForm) as the double-float apply
// (ok_apply_dd.cu) walks them: for each of four sums per site, a list of entries
//   sum += +-V w  or  +-V^dag w,   w = psi_s1 + unit psi_s2  of one neighbour,
// so that every product has one destination and no scalar.  Spins are 0, 1 = u, 2, 3 = l.  The sums of
// index w = 2 half + q are
//   D    temporal, two-hop and diagonal hops: half the output's components u_q, l_q;
//   S    nearest spatial hops: acc+_q, acc-_q (h+- = u +- l), stored halves;
//   O    on-site: A_q, B_q on u -+ i l.
#pragma once
#include "ok_internal.cuh"

namespace okgb {
namespace ddent {

// unit codes: 0 none, 1 + k: i^k
struct Entry {
  unsigned char m;      // colour matrix of the site record
  unsigned char hop;    // neighbour
  unsigned char flags;  // bit 0: adjoint of the matrix at the neighbour (else the matrix at x); bit 1: minus
  unsigned char src;    // s1 | s2 << 2 | unit << 4
};
constexpr int N_TWO = 6, N_D = 23, N_S = 35, N_ALL = 37;  // ends of: two-hop, D, S, O
constexpr int HOPS = 27, ON_SITE = 26;
struct Table {
  Entry e[4][N_ALL];
  signed char d[HOPS][4];
};

inline Table build() {
  Table t{};
  int nh = 0;
  auto hop = [&](int x, int y, int z, int w) {
    t.d[nh][0] = (signed char)x; t.d[nh][1] = (signed char)y; t.d[nh][2] = (signed char)z; t.d[nh][3] = (signed char)w;
    return nh++;
  };
  int ne[4] = {0, 0, 0, 0};
  auto put = [&](int w, int m, int h, bool adj, bool minus, int s1, int s2 = 0, int unit = -1) {  // unit = k of i^k
    t.e[w][ne[w]++] = Entry{(unsigned char)m, (unsigned char)h, (unsigned char)((adj ? 1 : 0) | (minus ? 2 : 0)),
                            (unsigned char)(s1 | s2 << 2 | (unit < 0 ? 0 : 1 + (unit & 3)) << 4)};
  };
  // sigma_k[q][q'] = i^u with q' and u
  auto sigma = [](int k, int q, int& qp, int& u) {
    qp = k == 2 ? q : 1 - q;
    u = k == 0 ? 0 : k == 1 ? (q ? 1 : 3) : (q ? 2 : 0);
  };
  auto dir3 = [](int I, int n, int (&d)[3]) { d[0] = n * (I == 0); d[1] = n * (I == 1); d[2] = n * (I == 2); };
  // two-hop: D_hq += (a psi_hq +- b sigma_I psi_{1-h}) through V; the entry's unit carries the sign of b
  for (int I = 0; I < 3; ++I)
    for (int b = 0; b < 2; ++b) {
      int d[3];
      dir3(I, b ? -2 : 2, d);
      const int h = hop(d[0], d[1], d[2], 0);
      for (int w = 0; w < 4; ++w) {
        int qp, u;
        sigma(I, w & 1, qp, u);
        put(w, M_VII + I, h, b, false, w, 2 * (1 - (w >> 1)) + qp, u + (b ? 2 : 0));
      }
    }
  // temporal: [[0, S], [S, -U]] forward, [[-U^dag, -S^dag], [-S^dag, 0]] backward, S = [[s3, n1], [n2, -s3]]
  {
    const int f = hop(0, 0, 0, 1), b = hop(0, 0, 0, -1);
    for (int w = 0; w < 4; ++w) {
      const int q = w & 1, o = 2 * (1 - (w >> 1));  // the other half's spins o, o + 1
      put(w, M_ST, f, false, q, o + q);
      put(w, M_ST + 1 + q, f, false, false, o + 1 - q);
      if (w >= 2) put(w, M_UT, f, false, true, w);
      put(w, M_ST, b, true, !q, o + q);
      put(w, M_ST + 2 - q, b, true, true, o + 1 - q);
      if (w < 2) put(w, M_UT, b, true, true, w);
    }
  }
  // diagonal: (sigma_I + sj sigma_J) from the other half through V (sj = 1) or X (sj = -1), minus the adjoint backward
  for (int P = 0; P < 3; ++P) {
    const int I = P == 2 ? 1 : 0, J = P == 0 ? 1 : 2;
    for (int form = 0; form < 2; ++form)
      for (int b = 0; b < 2; ++b) {
        const int st = b ? -1 : 1, sj = form ? -1 : 1;
        int d[3] = {0, 0, 0};
        d[I] += st;
        d[J] += st * sj;
        const int h = hop(d[0], d[1], d[2], 0);
        for (int w = 0; w < 4; ++w) {
          int qi, ui, qj, uj;
          sigma(I, w & 1, qi, ui);
          sigma(J, w & 1, qj, uj);
          if (sj < 0) uj += 2;
          const int o = 2 * (1 - (w >> 1));
          // i^ui psi_qi + i^uj psi_qj: the one with a real unit first, its sign taken out
          const bool swap = (ui & 1) != 0;
          const int s1 = swap ? qj : qi, s2 = swap ? qi : qj;
          const int u1 = swap ? uj : ui, u2 = swap ? ui : uj;   // u1 is 0 or 2 (sigma_x or sigma_z)
          put(w, (form ? M_XIJ : M_VIJ) + P, h, b, (b != 0) != ((u1 & 2) != 0), o + s1, o + s2, u2 - u1 + 4);
        }
      }
  }
  // spatial: acc_h q += block (q, r) of P_h on h_r forward, block (r, q)^dag of P_{1-h} backward
  for (int I = 0; I < 3; ++I)
    for (int b = 0; b < 2; ++b) {
      int d[3];
      dir3(I, b ? -1 : 1, d);
      const int h = hop(d[0], d[1], d[2], 0);
      for (int w = 0; w < 4; ++w)
        for (int r = 0; r < 2; ++r) {
          const int hh = w >> 1, q = w & 1;
          put(w, M_WP + 8 * I + 4 * (b ? 1 - hh : hh) + (b ? 2 * r + q : 2 * q + r), h, b, false, r, 2 + r, hh ? 2 : 0);
        }
    }
  // on-site: Y+ on u - i l (A), Y- on u + i l (B), Y = [[y3, y1], [y2, -y3]]
  {
    const int h = hop(0, 0, 0, 0);
    for (int w = 0; w < 4; ++w) {
      const int hh = w >> 1, q = w & 1, y = hh ? M_Y0M : M_Y0P, u = hh ? 1 : 3;
      put(w, y, h, false, q, q, 2 + q, u);
      put(w, y + 1 + q, h, false, false, 1 - q, 3 - q, u);
    }
  }
  return t;
}

}  // namespace ddent
}  // namespace okgb
