// Internal entry points of the even-odd preconditioned operator (Sec. 4), shared by the
// W_eo / D_hat code and the mass reweighting.  "Half vectors" hold the sites of one parity only
// ((t + z + y + x) mod 2): N_s / 2 sites in the site-tiled layout, site j = s / 2 of the doubled
// lattice.  All calls are asynchronous on the lattice's stream.
#pragma once
#include "dslash.cuh"
#include "qs_internal.cuh"

// inv = (4 + m0 + A)^-1 on the odd physical sites, [2][6][6][V_phys / 2] complex, the odd
// physical site p at index p / 2
int qs_clover_inverse_odd(qs_lattice *lat, double m0, double2 *inv);

// canonical full-lattice vectors -> half vectors of one parity
int qs_parity_pack(qs_lattice *lat, const double *in, double *out, int nrhs, int parity);
// the sites of one parity of canonical full-lattice vectors x = a - b (b may be NULL: a)
int qs_parity_unpack(qs_lattice *lat, const double *a, const double *b, double *x, int nrhs, int parity);

// out_o = f (D_oo)^-1 (D_oe in_e) (hop = 1), or f (D_oo)^-1 in_o (hop = 0), on half vectors; live:
// NULL or per right-hand side, 0 skips it
int qs_hat_odd(qs_lattice *lat, const double2 *inv, const double *in, double *out, int nrhs, int hop, double f,
               const int *live = nullptr);
// out_e = D_eo v_o + sigma add_e (half vectors)
int qs_hat_hop_even(qs_lattice *lat, const double *v, const double *add, double sigma, double *out, int nrhs);
// out = D_hat in (gamma5 = 1: Q_hat in) + sigma add on half vectors, inv from
// qs_clover_inverse_odd at the same m0; work: one half vector per right-hand side.  add may be
// NULL; part != NULL (with add): part[r][tile] gets the shares of Re (add_r, out_r) of the
// qs_hat_tiles() tiles.  in, add and work must not overlap out.
int qs_dhat_run(qs_lattice *lat, double m0, const double *in, double *out, int nrhs, int gamma5, double *work,
                const double2 *inv, const int *live = nullptr, const double *add = nullptr, double sigma = 0.0,
                double *part = nullptr);
int64_t qs_hat_tiles(const Geom &g);
