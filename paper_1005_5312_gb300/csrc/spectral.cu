// Spectral tables of the two kinds of photons that are not monochromatic.
//
// Blackbody point sources (Section 3.1.1's sources with the photoionisation
// and photoheating integrals of Appendix A): with u = nu / nu_L, the photon
// spectrum w(u) = u^2 / (e^(a u) - 1), a = h nu_L / (k T_eff), and the
// hydrogenic cross-section sigma_nu = sigma_L u^-3, a ray of Lyman-limit
// optical depth tau delivers per emitted ionising photon
//   F_ion(tau)  = int w u^-3 e^(-tau u^-3) du / int w du          (u >= 1)
//   F_heat(tau) = int w u^-3 (u - 1) e^(-tau u^-3) du / int w du
// so Gamma_eff = sum L F_ion / (4 pi r^2) (k_ion = sigma_L Gamma_eff) and the
// heating per neutral atom is sigma_L h nu_L sum L F_heat / (4 pi r^2).
//
// Recombination photons of the diffuse case (Section 4.1) spread evenly over
// the band 1 <= u <= 1 + D, D = k T_rec / (h nu_L):
//   R_ion(tau)  = (1/D) int u^-3 e^(-tau u^-3) du
//   R_heat(tau) = (1/D) int (u - 1) u^-3 e^(-tau u^-3) du
// in the same roles (Eq. gother for the heating).
//
// Each integral is tabulated as ln F on a grid in s = ln(1 + tau / tau0), by
// composite 6-point Gauss-Legendre (the blackbody over u in [1, 1 + 80/a], beyond
// which the spectrum is below e^-80 of its peak) in FP64, a thread per grid
// point that takes the nodes in order (on the host the 12.6 million exponentials
// of a blackbody held up the first solve with a new temperature for 38 ms,
// against 1.4 ms); the per-pair reduction interpolates linearly in s.
#include <math.h>

#include <vector>

#include "common.cuh"

namespace st {

namespace {
constexpr double kHnuL = kHnuLErg;
constexpr double kBoltz = kBoltzErg;
constexpr int kPanels = 256;
const double kGx[6] = {-0.9324695142031521, -0.6612093864662645, -0.2386191860831909,
                       0.2386191860831909,  0.6612093864662645,  0.9324695142031521};
const double kGw[6] = {0.1713244923791704, 0.3607615730481386, 0.4679139345726910,
                       0.4679139345726910, 0.3607615730481386, 0.1713244923791704};

// nodes and weights of composite Gauss-Legendre over [lo, hi]
void gl_nodes(double lo, double hi, int panels, std::vector<double> &x, std::vector<double> &w)
{
    const double hw = 0.5 * (hi - lo) / panels;
    for (int p = 0; p < panels; ++p) {
        double mid = lo + (2 * p + 1) * hw;
        for (int k = 0; k < 6; ++k) {
            x.push_back(mid + hw * kGx[k]);
            w.push_back(kGw[k] * hw);
        }
    }
}
}  // namespace

// ln of the two integrals of a spectrum given by its n quadrature nodes (weight
// w_j and u_j, then u_j^-3), normalised by z, at every grid point; into tab[0, kSpecN)
// and tab[kSpecN, 2 kSpecN).
__global__ void __launch_bounds__(64) k_spectral_table(const double *w, const double *u,
                                                       const double *iu3, int n, double z,
                                                       double ds, float *tab)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kSpecN) return;
    const double tau = kSpecTau0 * expm1(k * ds);
    double fi = 0.0, fh = 0.0;
    for (int j = 0; j < n; ++j) {
        const double v = w[j] * iu3[j] * exp(-tau * iu3[j]);
        fi += v;
        fh += v * (u[j] - 1.0);
    }
    tab[k] = (float)log(fmax(fi / z, 1e-300));
    tab[kSpecN + k] = (float)log(fmax(fh / z, 1e-300));
}

// Tabulates a spectrum of nodes (u, w) with normalisation z at tab (device).
static int tabulate(start_ctx *c, const std::vector<double> &u, const std::vector<double> &w,
                    double z, float *tab)
{
    const size_t n = u.size();
    std::vector<double> nodes(3 * n);
    for (size_t j = 0; j < n; ++j) {
        nodes[j] = w[j];
        nodes[n + j] = u[j];
        nodes[2 * n + j] = 1.0 / (u[j] * u[j] * u[j]);
    }
    DBuf buf;
    if (ensure(buf, nodes.size() * sizeof(double)))
        return set_err(c, START_ENOMEM, "out of device memory (spectral tables)");
    cudaError_t e = cudaMemcpyAsync(buf.p, nodes.data(), nodes.size() * sizeof(double),
                                    cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) {
        const double *d = buf.as<double>();
        const double ds = log1p(kSpecTauMax / kSpecTau0) / (kSpecN - 1);
        k_spectral_table<<<grid_for(kSpecN, 64), 64, 0, c->stream>>>(d, d + n, d + 2 * n, (int)n,
                                                                      z, ds, tab);
        ++c->launches;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);   // nodes are on the host
    }
    release(buf);   // stream-ordered
    return cuda_check(c, e, "k_spectral_table");
}

int spectral_table(start_ctx *c)
{
    const double T = c->p.T_eff, Tr = c->p.T_rec;
    if (c->spec_T == T && c->spec_Trec == Tr && c->spec_tab.p) return START_OK;
    c->spec_T = c->spec_Trec = -1.0;
    ST_TRY(ensure(c->spec_tab, 4 * kSpecN * sizeof(float)));
    float *tab = c->spec_tab.as<float>();
    ST_CUDA(c, cudaMemsetAsync(tab, 0, 4 * kSpecN * sizeof(float), c->stream));
    if (T > 0.0) {
        const double a = kHnuL / (kBoltz * T);
        std::vector<double> u, w;
        gl_nodes(1.0, 1.0 + 80.0 / a, kPanels, u, w);
        double z = 0.0;
        for (size_t j = 0; j < u.size(); ++j) {
            w[j] *= u[j] * u[j] / expm1(a * u[j]);
            z += w[j];
        }
        ST_TRY(tabulate(c, u, w, z, tab));
    }
    if (Tr > 0.0) {
        const double D = kBoltz * Tr / kHnuL;
        std::vector<double> u, w;
        gl_nodes(1.0, 1.0 + D, 16, u, w);
        ST_TRY(tabulate(c, u, w, D, tab + 2 * kSpecN));
    }
    c->spec_T = T;
    c->spec_Trec = Tr;
    return START_OK;
}

}  // namespace st
