// cheb_domain.h -- the interval s in [0, S] on which the embedding nets run as
// Chebyshev series (embed_cheb.cu); rows with s > S, pairs nearer than 1 / S,
// evaluate the net.
#pragma once

// S = 4/3, r = 0.75, where the cut-off is that of a model in A or Bohr (3 and
// more; below the O-H bond; S = 2 takes 24 terms instead of 20), and eight times
// the inverse of a cut-off below 2, which is no distance in those units: the same
// part of the rows for the same model in nm or m.  With 4/3 there every row is
// beyond S: 12,288 water atoms in nm took 27.1 ms an evaluation, now 3.3, as in A.
inline double dp_cheb_domain(double rcut) { return rcut < 2.0 ? 8.0 / rcut : 4.0 / 3.0; }
