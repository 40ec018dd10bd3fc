// Resident step of quadrilateral meshes: host interface (kernel in selbm_flow2d.cuh).
#pragma once
#include "selbm_kernels.cuh"

namespace slb {

// a value and the number of its exchange: 8 bytes per 32 bits of the value, each written and read
// as one access
template <typename Real>
struct Packet {
  unsigned long long w[sizeof(Real) / 4];
};

template <typename Real>
struct Flow2DArgs {
  int E, Gs, epc, nsteps;
  int filter, pending, has_force;
  unsigned epoch;               // of the last exchange before this launch
  Real dt, half_dt, omega, rho0, g[3];
  const int32_t *l2g, *bslot;
  const uint8_t *owner;
  const Real *el_drdx, *el_J, *drdx, *wJ, *minv;
  const int *gexp;              // FP64, curved: metrics are taken times 2^gexp[e]
  const WallPt<Real> *walls;
  const int32_t *wall_off;
  const Real *wall_u;
  const int32_t *loc_u;         // [E Nb] shared-node index of each local boundary node
  const int32_t *loc_off;       // [E Nb + 1] its copies, ascending, itself included, each as the index of a fetched
  const int32_t *loc_slot;      //   share of its CTA, or -3 - (local element Nb + slot) inside the CTA
  const int32_t *loc_base;      // [E Nb] the owner's copy: -1 itself, -3 - (local element Nb + slot), or fetched
  const int32_t *rem_off, *rem; // [CTAs + 1] trace offsets 9 Nb e' + b' of the shares a CTA fetches
  const int32_t *bas_off, *bas; // [CTAs + 1] shared-node indices of the owners' values a CTA fetches
  int rmax, bmax;               // most of them
  int *abort;                   // host memory: set when a wait gives up
  void *T;                      // [2][E][9][Nb] packets: shares
  void *base;                   // [Gb][10] packets: owner's f^0 and rho of shared nodes after a filter
  Real *f;                      // [9][Gs] state
};

// learned control of the resident step (see selbm_set_learned_filter)
template <typename Real>
struct Learn2DArgs {
  const __nv_bfloat16 *W;       // network parameters
  const Real *lo, *hi, *Vinv;   // [2n] training range; [n][n] nodal -> modal
  int *flag, *n_fallback;
  double *acc;                  // [2..4] mass, kinetic energy of the last pass, whether there was one
  Real *sigma_out;              // [E][n]
  Packet<double> *sums;         // [2][CTAs][2] packets: drift sums of a pass
  double mass_bound, ke_bound;
  int check_ke, pass;           // number of the first control pass of this launch
};

// probe: *fits = whether the SMs hold the mesh at p.epc elements a CTA; else launches p.nsteps steps
template <typename Real>
cudaError_t launch_flow2d(int N, bool affine, bool probe, const Flow2DArgs<Real> &p, const SplitHost &h,
                          const Learn2DArgs<Real> *lc, bool *fits, cudaStream_t s);

}  // namespace slb
