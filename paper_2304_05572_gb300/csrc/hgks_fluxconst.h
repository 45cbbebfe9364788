// hgks_fluxconst.h -- the constants of the gas-kinetic flux, formed once on the host.
#pragma once

namespace hgks {

// Kt = K + D - 1 counts the internal degrees of freedom as seen in the frame moving with the
// tangential velocity (2D: xi and the peculiar tangential velocity; 1D: xi alone).
struct FluxConst {
    double gm1, rgm1;      // gamma - 1, 1/(gamma - 1)
    double Kt, ktp2;       // Kt, Kt + 2
    double gq;             // (Kt + 3)/2: H = U^2/2 + gq h
    double k3, k6, hk6;    // Kt + 3, Kt + 6, (Kt + 6)/2
    double mu, c1, c2;
    double prfix;          // 1/Pr - 1 for viscous runs with Pr != 1, else 0
    int viscous, tau_zero;
};

inline FluxConst flux_const(double gm1, double Kt, double mu, double c1, double c2, double prfix, int viscous, int tau_zero)
{
    FluxConst f;
    f.gm1 = gm1; f.rgm1 = 1.0 / gm1;
    f.Kt = Kt; f.ktp2 = Kt + 2.0;
    f.gq = 0.5 * (Kt + 3.0);
    f.k3 = Kt + 3.0; f.k6 = Kt + 6.0; f.hk6 = 0.5 * (Kt + 6.0);
    f.mu = mu; f.c1 = c1; f.c2 = c2; f.prfix = prfix;
    f.viscous = viscous; f.tau_zero = tau_zero;
    return f;
}

}  // namespace hgks
