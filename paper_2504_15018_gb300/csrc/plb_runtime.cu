// C ABI of the P-LBM library (include/plb.h): handle management, workspace layout,
// host<->device staging, and the launch sequence of one time step.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "plb.h"
#include "plb_host.h"
#include "plb_launch.h"
#include "plb_plain.cuh"

namespace {
thread_local std::string g_err;
}  // namespace

namespace plb {
int set_error(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}
}  // namespace plb

namespace {
#define fail plb::set_error

#define PLB_CUDA(call)                                                                       \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) return fail(PLB_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

constexpr unsigned MAGIC = 0x504c4231u;   // "PLB1"
}  // namespace

namespace plb {

bool make_layout(int lattice, const int dims[3], int precision, Layout &L, int streaming) {
    if (lattice != PLB_D2Q9 && lattice != PLB_D3Q19) return false;
    if (precision < PLB_FP64 || precision > PLB_FP16S) return false;
    if (!dims || dims[0] < 1 || dims[1] < 1 || dims[2] < 1) return false;
    if (lattice == PLB_D2Q9 && dims[2] != 1) return false;
    L.Q = lattice == PLB_D2Q9 ? 9 : 19;
    L.D = lattice == PLB_D2Q9 ? 2 : 3;
    L.n = (long long)dims[0] * dims[1] * dims[2];
    if (L.n > (1LL << 40)) return false;
    L.s_pop = precision == PLB_FP64 ? 8 : (precision == PLB_FP32 ? 4 : 2);
    L.s_psi = precision == PLB_FP64 ? 8 : 4;
    L.pstride = (L.n + 127) / 128 * 128;
    L.gx = 16 / L.s_psi;
    L.px = (int)((dims[0] + 2 * L.gx + 31) / 32 * 32);
    L.py = dims[1] + 2;
    L.pz = L.D == 3 ? dims[2] + 2 : 1;
    L.psi_elems = (long long)L.px * L.py * L.pz;
    L.chunk = L.n < (1LL << 18) ? L.n : (1LL << 18);
    L.max_blocks = 1024;
    size_t off = 0;
    L.off_pops = off;
    off = align256(off + (size_t)L.Q * L.pstride * L.s_pop);
    L.off_pops2 = L.off_pops;
    if (streaming == PLB_STREAM_FUSED) {
        L.off_pops2 = off;
        off = align256(off + (size_t)L.Q * L.pstride * L.s_pop);
    }
    L.off_psi = off;
    off = align256(off + (size_t)L.psi_elems * L.s_psi);
    L.off_partials = off;
    off = align256(off + (size_t)L.max_blocks * 4 * sizeof(double));
    L.off_out = off;
    off = align256(off + kReduceOut * sizeof(double));
    L.off_staging = off;
    const int per_cell = L.Q > L.D + 2 ? L.Q : L.D + 2;
    // (a small lattice's staging area also serves as the second population copy of many-step launches)
    const size_t staged = (size_t)L.chunk * per_cell * sizeof(double), copy = (size_t)L.Q * L.pstride * L.s_pop;
    off = align256(off + (L.chunk == L.n && copy > staged ? copy : staged));
    L.off_flags = off;
    off = align256(off + 64);
    L.off_counts = off;
    off = align256(off + kTileWords * sizeof(unsigned));
    L.total = off;
    return true;
}

}  // namespace plb

namespace {

void reduce_final_launch(const double *partials, int nblocks, int is_max, const unsigned *flags, double *out,
                         cudaStream_t st);

const plb::Launchers *launchers_for(int lattice, int precision) {
    switch (precision) {
        case PLB_FP64: return plb::launchers_fp64(lattice);
        case PLB_FP32: return plb::launchers_fp32(lattice);
        default: return plb::launchers_fp16(lattice);
    }
}

void *pops_ptr(plb_t *h) { return h->pops; }
void *psi_ptr(plb_t *h) { return h->psi; }
double *staging_ptr(plb_t *h) { return h->staging; }

// Cells per staging chunk for a transfer of `need` FP64 values per cell (the staging area
// holds chunk x max(Q, D + 2) values).
long long stage_cells(const plb::Layout &L, int need) {
    const long long per_cell = L.Q > L.D + 2 ? L.Q : L.D + 2;
    const long long c = L.chunk * per_cell / need;
    return c < L.n ? c : L.n;
}

// Device address of a caller's buffer that kernels can access directly (device or managed
// memory, or pinned / registered host memory), else NULL (pageable host memory).
template <class T> T *device_view(T *ptr) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged || a.type == cudaMemoryTypeHost)
        return static_cast<T *>(a.devicePointer);
    return nullptr;
}

// Counters of the many-step launch: all tiles at the same count (also after a wait that gave up).
cudaError_t clear_counts(plb_t *h) {
    return h->counts ? cudaMemsetAsync(h->counts, 0, plb::kTileWords * sizeof(unsigned), h->stream) : cudaSuccess;
}

__global__ void k_forget_timeout(unsigned *flags) { atomicAnd(flags, ~(unsigned)plb::FLAG_TIMEOUT); }

// Before the populations are replaced: a wait that gave up is forgotten (the other flags stay).
cudaError_t forget_timeout(plb_t *h) {
    if (!h->counts) return cudaSuccess;
    k_forget_timeout<<<1, 1, 0, h->stream>>>(h->kp.flags);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : clear_counts(h);
}

int check_launch() {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(PLB_ECUDA, "kernel launch: %s", cudaGetErrorString(e));
    return PLB_OK;
}

}  // namespace

extern "C" {

const char *plb_last_error(void) { return g_err.c_str(); }

void plb_default_opts(plb_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->kappa = 1.0;
    o->tau_v = 0.0;
    o->collision = PLB_BGK;
    o->s_e = o->s_eps = o->s_q = o->s_pi = o->s_m = 1.0;
    o->precision = PLB_FP32;
    o->rho_ref = 0.0;
    o->wall_y = 0;
}

int plb_velocity_set(int lattice, int *c, double *w) {
    static const int c2[9][2] = {{0, 0}, {1, 0}, {-1, 0}, {0, 1}, {0, -1}, {1, 1}, {-1, -1}, {1, -1}, {-1, 1}};
    static const int c3[19][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0}, {0, 1, 0},  {0, -1, 0}, {0, 0, 1},  {0, 0, -1},
                                  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}, {1, 0, 1},  {-1, 0, -1}, {1, 0, -1},
                                  {-1, 0, 1}, {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
    if (lattice == PLB_D2Q9) {
        for (int i = 0; i < 9; ++i) {
            if (c) {
                c[3 * i] = c2[i][0];
                c[3 * i + 1] = c2[i][1];
                c[3 * i + 2] = 0;
            }
            if (w) w[i] = i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
        }
        return 9;
    }
    if (lattice == PLB_D3Q19) {
        for (int i = 0; i < 19; ++i) {
            if (c)
                for (int a = 0; a < 3; ++a) c[3 * i + a] = c3[i][a];
            if (w) w[i] = i == 0 ? 1.0 / 3.0 : (i < 7 ? 1.0 / 18.0 : 1.0 / 36.0);
        }
        return 19;
    }
    return -1;
}

size_t plb_workspace_bytes(int lattice, const int dims[3], const plb_opts *opts) {
    plb_opts o;
    plb_default_opts(&o);
    if (opts) o = *opts;
    plb::Layout L;
    if (!plb::make_layout(lattice, dims, o.precision, L, o.streaming)) return 0;
    return L.total;
}

int plb_solve_params(const plb_eos_params *eos, double *rho_v, double *rho_l, double *p0) {
    if (!eos) return fail(PLB_EINVAL, "eos is NULL");
    double rv = 0, rl = 0, pp = 0;
    int st = plb::solve_coexistence(*eos, rv, rl, pp);
    if (st != PLB_OK) return fail(st, "no liquid-vapour coexistence for these EOS parameters");
    if (rho_v) *rho_v = rv;
    if (rho_l) *rho_l = rl;
    if (p0) *p0 = pp;
    return PLB_OK;
}

int plb_si_convert(const double si[6], const double lat[3], double xi, double out[11]) {
    if (!si || !lat || !out) return fail(PLB_EINVAL, "NULL argument");
    int st = plb::si_convert(si, lat, xi, out);
    if (st != PLB_OK) return fail(st, "invalid physical or lattice inputs");
    return PLB_OK;
}

}  // extern "C"

namespace plb {

int check_create_args(int lattice, const int dims[3], const plb_eos_params *eos, double tau, double G, double eps,
                      const plb_opts *opts, plb_opts &o, Layout &lay) {
    if (!eos) return fail(PLB_EINVAL, "eos is NULL");
    plb_default_opts(&o);
    if (opts) o = *opts;
    if (o.streaming != PLB_STREAM_AA && o.streaming != PLB_STREAM_FUSED) return fail(PLB_EINVAL, "bad streaming");
    if (!make_layout(lattice, dims, o.precision, lay, o.streaming))
        return fail(PLB_EINVAL, "bad lattice, dims or precision");
    if (o.streaming == PLB_STREAM_FUSED &&
        (o.precision == PLB_FP64 || dims[0] % 2 != 0 || lay.n * lay.s_pop >= (1LL << 32)))
        return fail(PLB_EUNSUPPORTED, "fused streaming needs FP32 or FP16S storage, even nx and population planes "
                                      "below 4 GiB (< 2^30 cells FP32, < 2^31 FP16S)");
    if (!(tau > 0.5) || !std::isfinite(tau)) return fail(PLB_EINVAL, "tau must be > 1/2");
    if (!(G < 0.0) || !std::isfinite(G)) return fail(PLB_EINVAL, "G must be negative");
    if (!std::isfinite(eps) || !std::isfinite(o.kappa)) return fail(PLB_EINVAL, "eps and kappa must be finite");
    if (o.collision != PLB_BGK && o.collision != PLB_MRT) return fail(PLB_EINVAL, "bad collision");
    if (o.tau_v > 0.0 && !(o.tau_v > 0.5)) return fail(PLB_EINVAL, "tau_v must be > 1/2");
    if (o.fp16_rounding != 0 && o.fp16_rounding != 1) return fail(PLB_EINVAL, "fp16_rounding must be 0 or 1");
    if (o.wall_rho > 0.0 && !o.wall_y) return fail(PLB_EINVAL, "wall_rho needs walls (wall_y = 1)");
    if (!std::isfinite(o.wall_rho)) return fail(PLB_EINVAL, "wall_rho must be finite");
    if (eos->kind == PLB_EOS_PR) {
        if (!(eos->a > 0 && eos->b > 0 && eos->R > 0 && eos->T_over_Tc > 0)) return fail(PLB_EINVAL, "bad PR constants");
    } else if (eos->kind == PLB_EOS_PAPER) {
        if (!(eos->rho_v > 0 && eos->rho_l > eos->rho_v && eos->pc_over_rhoc3 > 0))
            return fail(PLB_EINVAL, "bad paper-EOS constants");
    } else {
        return fail(PLB_EINVAL, "unknown EOS kind");
    }
    if (!(eos->p_scale >= 0.0)) return fail(PLB_EINVAL, "p_scale must be >= 0");
    return PLB_OK;
}

bool needs_coexistence(double tau, const plb_opts &o) {
    return (o.precision == PLB_FP16S && !(o.rho_ref > 0)) ||
           (o.tau_v > 0.0 && o.tau_v != tau && !(o.tau_rho_l > o.tau_rho_v));
}

int fill_kparams(const int dims[3], const plb_eos_params &eos, double tau, double G, double eps, const plb_opts &o,
                 const Layout &lay, double rv, double rl, KParams &k) {
    std::memset(&k, 0, sizeof(k));
    k.nx = dims[0];
    k.ny = dims[1];
    k.nz = dims[2];
    k.z0 = 0;
    k.nzl = dims[2];
    k.n = lay.n;
    k.pstride = lay.pstride;
    k.wall_y = o.wall_y ? 1 : 0;
    k.wall_fixed = (o.wall_y && o.wall_rho > 0.0) ? 1 : 0;
    k.px = lay.px;
    k.py = lay.py;
    k.psi_origin = lay.gx + (long long)lay.px * (1 + (long long)lay.py * (lay.D == 3 ? 1 : 0));
    Phys<double> &d = k.d;
    d.G = G;
    d.inv_G = 1.0 / G;
    // Eq. interactionForce with the eps coefficient that realises Eq. New_Pressure_Tensor.
    d.A_m1m2 = -(G / 12.0) * (2.0 * o.kappa - 2.0 - 3.0 * eps);
    d.B_m1tr = (G / 6.0) * (o.kappa - 1.0);
    d.tau_l = tau;
    d.om_const = 1.0 / tau;
    k.var_tau = o.tau_v > 0.0 && o.tau_v != tau;
    d.tau_v = k.var_tau ? o.tau_v : tau;
    double trv = o.tau_rho_v, trl = o.tau_rho_l;
    if (k.var_tau && !(trl > trv)) {
        trv = rv;
        trl = rl;
        if (!(trl > trv))
            return fail(PLB_EINVAL, "tau(rho) needs tau_rho_l > tau_rho_v (EOS has no coexistence to default to)");
    }
    d.tau_rho_v = trv;
    d.inv_drho_tau = k.var_tau ? 1.0 / (trl - trv) : 0.0;
    d.s_rate[0] = 0.0;
    d.s_rate[1] = o.s_e;
    d.s_rate[2] = o.s_eps;
    d.s_rate[3] = o.s_q;
    d.s_rate[4] = o.s_pi;
    d.s_rate[5] = o.s_m;
    for (int a = 0; a < 3; ++a) d.fext[a] = a < lay.D ? o.body_force[a] : 0.0;
    d.rho_ref = o.precision == PLB_FP16S ? (o.rho_ref > 0 ? o.rho_ref : rv) : 0.0;
    k.eos_kind = eos.kind;
    if (eos.kind == PLB_EOS_PR) {
        const PrConstants c = pr_constants(eos);
        d.pr_RT = c.RT;
        d.pr_b = eos.b;
        d.pr_aalpha = c.aalpha;
    } else {
        d.pe_P = eos.pc_over_rhoc3;
        d.pe_rv = eos.rho_v;
        d.pe_rl = eos.rho_l;
        d.pe_sv = std::sqrt(eos.rho_v);
    }
    d.p_scale = eos.p_scale;
    // constants of the plain FP64 evaluation, each rounded as its expression is written
    PlainPhys &pl = k.pl;
    if (eos.kind == PLB_EOS_PR) {
        const double Tc = 0.0778 * eos.a / (0.45724 * eos.b * eos.R);
        const double T = eos.T_over_Tc * Tc;
        const double m = 0.37464 + 1.54226 * eos.omega - 0.26992 * eos.omega * eos.omega;
        const double g = 1.0 + m * (1.0 - std::sqrt(T / Tc));
        pl.R = eos.R;
        pl.T = T;
        pl.b = eos.b;
        pl.a_alpha = eos.a * (g * g);
    } else {
        const double sv = std::sqrt(eos.rho_v);
        pl.P = eos.pc_over_rhoc3;
        pl.rv_2rl = eos.rho_v - 2.0 * eos.rho_l;
        pl.sv3 = 3.0 * sv;
        pl.sv2rl = 2.0 * sv * eos.rho_l;
        pl.svrlrl = sv * eos.rho_l * eos.rho_l;
    }
    pl.p_scale = eos.p_scale;
    pl.G = G;
    pl.K1 = (G / 12.0) * (-3.0 * eps + 2.0 * o.kappa - 2.0);
    pl.K2 = (G / 6.0) * (o.kappa - 1.0);
    pl.tau_l = tau;
    pl.tau_v = d.tau_v;
    pl.tau_rho_v = trv;
    pl.d_rho = trl - trv;
    pl.d_tau = tau - d.tau_v;
    for (int r = 0; r < 6; ++r) {
        pl.s_rate[r] = d.s_rate[r];
        pl.s_half[r] = 1.0 - d.s_rate[r] / 2.0;
    }
    pl.inv_G = plain::reciprocal(G);
    pl.inv_tau = plain::reciprocal(tau);
    pl.inv_d_rho = k.var_tau ? plain::reciprocal(pl.d_rho) : Recip{0.0, 0.0};
    for (int a = 0; a < 3; ++a) pl.fext[a] = d.fext[a];
    if (k.wall_fixed) {
        // Eq. Interaction_Potential at the wall density
        const double arg = plain::psi_arg(pl, eos.kind, o.wall_rho);
        if (!(arg >= 0.0)) return fail(PLB_EINVAL, "psi is not defined at wall_rho for this EOS");
        d.psi_wall = std::sqrt(arg);
    }
    k.stochastic = o.precision == PLB_FP16S && o.fp16_rounding == 1;
    k.salt = 0;
    // FP32 copy (rounded once here, not per thread)
    Phys<float> &f = k.f;
    const double *src = reinterpret_cast<const double *>(&d);
    float *dst = reinterpret_cast<float *>(&f);
    static_assert(sizeof(Phys<double>) == 2 * sizeof(Phys<float>), "Phys layout");
    for (size_t m = 0; m < sizeof(Phys<double>) / sizeof(double); ++m) dst[m] = (float)src[m];
    return PLB_OK;
}

const Launchers *launchers_for_precision(int lattice, int precision) { return launchers_for(lattice, precision); }

}  // namespace plb

extern "C" {

int plb_create(int lattice, const int dims[3], const plb_eos_params *eos, double tau, double G, double eps,
               const plb_opts *opts, void *dev_workspace, size_t ws_bytes, void *cuda_stream, plb_t **out) {
    if (!out) return fail(PLB_EINVAL, "out is NULL");
    *out = nullptr;
    plb_opts o;
    plb::Layout lay;
    int st = plb::check_create_args(lattice, dims, eos, tau, G, eps, opts, o, lay);
    if (st != PLB_OK) return st;
    if (!dev_workspace) return fail(PLB_EINVAL, "workspace is NULL");
    if (reinterpret_cast<uintptr_t>(dev_workspace) % 256 != 0) return fail(PLB_EINVAL, "workspace not 256-byte aligned");
    if (ws_bytes < lay.total)
        return fail(PLB_ENOMEM, "workspace has %zu bytes, needs %zu", ws_bytes, lay.total);

    plb_t *h = new plb_state();
    h->lattice = lattice;
    std::memcpy(h->dims, dims, sizeof(h->dims));
    h->opts = o;
    h->eos = *eos;
    h->tau = tau;
    h->G = G;
    h->eps = eps;
    h->lay = lay;
    h->ws = static_cast<char *>(dev_workspace);
    h->pops = h->ws + lay.off_pops;
    h->pops2 = o.streaming == PLB_STREAM_FUSED ? h->ws + lay.off_pops2 : nullptr;
    h->psi = h->ws + lay.off_psi;
    h->partials = reinterpret_cast<double *>(h->ws + lay.off_partials);
    h->out = reinterpret_cast<double *>(h->ws + lay.off_out);
    h->staging = reinterpret_cast<double *>(h->ws + lay.off_staging);
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    h->t = 0;
    h->odd = 0;
    h->L = launchers_for(lattice, o.precision);
    // Coexistence densities: defaults for the tau interpolation and the FP16 shift.
    double rv = 0, rl = 0, pp = 0;
    if (plb::solve_coexistence(*eos, rv, rl, pp) != PLB_OK) {
        rv = rl = pp = 0;
    }
    h->rho_v = rv;
    h->rho_l = rl;
    h->p0 = pp;
    plb::KParams &k = h->kp;
    st = plb::fill_kparams(dims, *eos, tau, G, eps, o, lay, rv, rl, k);
    if (st != PLB_OK) {
        delete h;
        return st;
    }
    h->opts.rho_ref = k.d.rho_ref;
    k.flags = reinterpret_cast<unsigned *>(h->ws + lay.off_flags);
    h->counts = reinterpret_cast<unsigned *>(h->ws + lay.off_counts);
    cudaError_t e = cudaMemsetAsync(h->psi, 0, (size_t)lay.psi_elems * lay.s_psi, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(k.flags, 0, 64, h->stream);
    if (e == cudaSuccess) e = clear_counts(h);
    if (e == cudaSuccess && k.wall_fixed) {
        h->L->wall_fill(k, h->psi, h->stream);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        delete h;
        return fail(PLB_ECUDA, "workspace set-up: %s", cudaGetErrorString(e));
    }
    *out = h;
    return PLB_OK;
}

void plb_destroy(plb_t *h) {
    if (h && !h->view) delete h;
}

long long plb_time(const plb_t *h) { return h ? h->t : -1; }

int plb_init(plb_t *h, const double *rho0, const double *u0) {
    if (h && h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: use plb_batch_init");
    return plb::init_state(h, rho0, u0);
}

int plb_init_physical(plb_t *h, const double *rho0, const double *u0) {
    if (h && h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: use plb_batch_init_physical");
    const int st = plb::init_state(h, rho0, u0);
    return st != PLB_OK ? st : plb::rebalance_state(h);
}

}  // extern "C"

int plb::init_state(plb_state *h, const double *rho0, const double *u0) {
    if (!h || !rho0) return fail(PLB_EINVAL, "NULL argument");
    const long long n = h->lay.n;
    // rho0 and u0 are checked on the device as k_init reads them (a host scan of 33 M values
    // costs tens of milliseconds): flags cleared, first-invalid-index slots set to all ones
    PLB_CUDA(cudaMemsetAsync(h->kp.flags, 0, 64, h->stream));
    PLB_CUDA(cudaMemsetAsync(h->kp.flags + plb::FLAG_SLOT_RHO, 0xff, 16, h->stream));
    PLB_CUDA(clear_counts(h));
    const double *drho0 = device_view(rho0), *du0 = u0 ? device_view(u0) : nullptr;
    if (drho0 && (!u0 || du0)) {
        // inputs the device can read: one launch over all cells
        h->L->init(h->kp, pops_ptr(h), drho0, du0, 0, n, h->stream);
        int st = check_launch();
        if (st) return st;
    }
    double *stg = staging_ptr(h);
    const long long chunk = stage_cells(h->lay, 1 + (u0 ? h->lay.D : 0));
    for (long long c0 = (drho0 && (!u0 || du0)) ? n : 0; c0 < n; c0 += chunk) {
        const long long cn = (n - c0) < chunk ? (n - c0) : chunk;
        PLB_CUDA(cudaMemcpyAsync(stg, rho0 + c0, cn * sizeof(double), cudaMemcpyHostToDevice, h->stream));
        if (u0)
            for (int a = 0; a < h->lay.D; ++a)
                PLB_CUDA(cudaMemcpyAsync(stg + (1 + a) * cn, u0 + a * n + c0, cn * sizeof(double),
                                         cudaMemcpyHostToDevice, h->stream));
        h->L->init(h->kp, pops_ptr(h), stg, u0 ? stg + cn : nullptr, c0, cn, h->stream);
        int st = check_launch();
        if (st) return st;
    }
    unsigned long long w[3];        // flag word, first invalid rho0 index, first invalid u0 index
    PLB_CUDA(cudaMemcpyAsync(w, h->kp.flags, sizeof(w), cudaMemcpyDeviceToHost, h->stream));
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    h->t = 0;
    h->odd = 0;
    if ((unsigned)w[0] & plb::FLAG_BAD_INPUT) {
        PLB_CUDA(cudaMemsetAsync(h->kp.flags, 0, 64, h->stream));
        if (w[1] != ~0ull) return fail(PLB_EINVAL, "rho0[%lld] is not a positive number", (long long)w[1]);
        return fail(PLB_EINVAL, "u0[%lld] is not finite", (long long)w[2]);
    }
    return PLB_OK;
}

int plb::rebalance_state(plb_state *h) {
    h->L->psi(h->kp, pops_ptr(h), psi_ptr(h), 0, h->stream);
    int st = check_launch();
    if (st) return st;
    h->L->rebalance(h->kp, pops_ptr(h), psi_ptr(h), h->stream);
    return check_launch();
}

namespace {

// Steps of one launch: a launch holds its SMs to its end, so a longer call is several launches, of about a
// millisecond each (an FP64 cell costs some eight times an FP32 one), between which the work of other
// streams gets its turn.  A launch's start (some 10 us) is then a hundredth of it.
int tile_steps(const plb_t *h) {
    const long long cells = h->opts.precision == PLB_FP64 ? 1LL << 21 : 1LL << 24;
    const long long steps = cells / h->lay.n;
    return steps < 16 ? 16 : (steps > 512 ? 512 : (int)(steps & ~1LL));
}

// Advances a small lattice by as many of n steps as many-step launches take (taken; 0: none).  In-place
// lattices borrow the staging area as the second population copy, take an even number of steps (the
// populations end where they were) and start at even parity.
int step_tiles(plb_t *h, int n, int coll, int &taken) {
    const int form = h->pops2 ? 1 : 0;
    taken = 0;
    if (h->tiles_state == 0) {
        const plb::Layout &L = h->lay;
        bool use = h->counts && L.n == L.chunk;        // the staging area holds a second copy
        if (use) use = h->L->tile_plan[form](h->kp, coll, h->tiles);
        h->tiles_state = use ? 1 : -1;
    }
    if (h->tiles_state < 0) return PLB_OK;
    if (!h->pops2 && h->odd) {
        // one in-place step brings the natural layout back
        if (n < h->tiles.least + 1) return PLB_OK;
        h->kp.salt = (unsigned)h->t;
        h->L->psi(h->kp, h->pops, h->psi, 1, h->stream);
        h->L->collide[coll](h->kp, h->pops, h->psi, 1, h->stream);
        h->odd = 0;
        h->t += 1;
        taken = 1;
        const int st = check_launch();                 // (before the error of a launch of tiles is dropped)
        if (st != PLB_OK) return st;
    }
    const int most = tile_steps(h);
    while (n - taken >= h->tiles.least) {
        plb::TileArgs t = h->tiles;
        t.nsteps = n - taken < most ? n - taken : most;
        if (!h->pops2) t.nsteps &= ~1;
        t.a = h->pops;
        t.b = h->pops2 ? h->pops2 : reinterpret_cast<char *>(h->staging);
        t.counts = h->counts;
        t.spin_limit = h->withhold ? h->withhold : 1u << 22;       // about 0.7 s of polling
        t.withhold = h->withhold ? 1 : 0;
        h->withhold = 0;
        h->kp.salt = (unsigned)h->t;
        cudaError_t e = h->L->tile_run[form](h->kp, coll, t, h->stream);
        if (e != cudaSuccess) {
            // the tiles do not fit this context (fewer SMs than the device reports): the other kernels do
            cudaGetLastError();
            h->tiles_state = -1;
            return PLB_OK;
        }
        if (h->pops2 && (t.nsteps & 1)) std::swap(h->pops, h->pops2);
        h->t += t.nsteps;
        h->many_launches += 1;
        h->many_steps += t.nsteps;
        taken += t.nsteps;
    }
    return PLB_OK;
}

}  // namespace

extern "C" {

int plb_step(plb_t *h, int n) {
    if (!h || n < 0) return fail(PLB_EINVAL, "bad argument");
    if (h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: use plb_batch_step");
    if (h->slab) return fail(PLB_EINVAL, "this lattice is a slab: step it with plb_slab_pass and plb_slab_exchange");
    const int coll = h->opts.collision == PLB_MRT ? 1 : 0;
    int taken = 0;
    const int st = step_tiles(h, n, coll, taken);
    if (st != PLB_OK) return st;
    n -= taken;
    if (h->pops2) {
        // single pass: read the current copy, push into the other, swap
        for (int k = 0; k < n; ++k) {
            h->kp.salt = (unsigned)h->t;
            h->L->fused[coll](h->kp, h->pops, h->pops2, h->stream);
            std::swap(h->pops, h->pops2);
            h->t += 1;
        }
        return check_launch();
    }
    for (int k = 0; k < n; ++k) {
        h->kp.salt = (unsigned)h->t;
        h->L->psi(h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
        h->L->collide[coll](h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
        h->odd ^= 1;
        h->t += 1;
    }
    return check_launch();
}

int plb_withhold_counts(plb_t *h, unsigned spin_limit) {
    if (!h) return fail(PLB_EINVAL, "NULL handle");
    h->withhold = spin_limit;
    return PLB_OK;
}

int plb_launch_counts(const plb_t *h, long long counts[2]) {
    if (!h || !counts) return fail(PLB_EINVAL, "NULL argument");
    counts[0] = h->many_launches;
    counts[1] = h->many_steps;
    return PLB_OK;
}

int plb_step_timed(plb_t *h, int n, double ms[2]) {
    if (!h || n < 0 || !ms) return fail(PLB_EINVAL, "bad argument");
    if (h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: use plb_batch_step");
    if (h->slab) return fail(PLB_EINVAL, "this lattice is a slab: step it with plb_slab_pass and plb_slab_exchange");
    ms[0] = ms[1] = 0.0;
    if (n == 0) return PLB_OK;
    const int coll = h->opts.collision == PLB_MRT ? 1 : 0;
    std::vector<cudaEvent_t> ev(2 * (size_t)n + 1);
    for (auto &e : ev) PLB_CUDA(cudaEventCreate(&e));
    int st = PLB_OK;
    PLB_CUDA(cudaEventRecord(ev[0], h->stream));
    for (int k = 0; k < n; ++k) {
        h->kp.salt = (unsigned)h->t;
        if (h->pops2) {
            // one kernel per step: it is reported as the fused pass, the psi interval is empty
            cudaEventRecord(ev[2 * k + 1], h->stream);
            h->L->fused[coll](h->kp, h->pops, h->pops2, h->stream);
            cudaEventRecord(ev[2 * k + 2], h->stream);
            std::swap(h->pops, h->pops2);
            h->t += 1;
            continue;
        }
        h->L->psi(h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
        cudaEventRecord(ev[2 * k + 1], h->stream);
        h->L->collide[coll](h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
        cudaEventRecord(ev[2 * k + 2], h->stream);
        h->odd ^= 1;
        h->t += 1;
    }
    st = check_launch();
    cudaError_t e = cudaEventSynchronize(ev[2 * n]);
    for (int k = 0; k < n && e == cudaSuccess; ++k) {
        float a = 0, b = 0;
        cudaEventElapsedTime(&a, ev[2 * k], ev[2 * k + 1]);
        cudaEventElapsedTime(&b, ev[2 * k + 1], ev[2 * k + 2]);
        ms[0] += a;
        ms[1] += b;
    }
    for (auto &x : ev) cudaEventDestroy(x);
    if (e != cudaSuccess) return fail(PLB_ECUDA, "cudaEventSynchronize: %s", cudaGetErrorString(e));
    return st;
}

static int status_of(unsigned flags) {
    if (flags & plb::FLAG_TIMEOUT) return fail(PLB_ETIMEOUT, "a device-side wait of a step gave up");
    if (flags & plb::FLAG_NONFINITE) return fail(PLB_ENONFINITE, "a density became non-positive or non-finite");
    if (flags & plb::FLAG_PSI_DOMAIN) return fail(PLB_EPSI_DOMAIN, "2 (p_EOS - rho/3) / G < 0 on some cell");
    return PLB_OK;
}

int plb_status(plb_t *h) {
    if (!h) return fail(PLB_EINVAL, "NULL handle");
    unsigned flags = 0;
    PLB_CUDA(cudaMemcpyAsync(&flags, h->kp.flags, sizeof(unsigned), cudaMemcpyDeviceToHost, h->stream));
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    return status_of(flags);
}

int plb_moments(plb_t *h, double *rho, double *u, double *p) {
    if (!h) return fail(PLB_EINVAL, "NULL handle");
    h->L->psi(h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
    const int D = h->lay.D;
    const long long n = h->lay.n, chunk = stage_cells(h->lay, D + 2);
    // Outputs the device can write (device memory, or host memory the runtime has pinned or
    // registered): one launch writes them directly; otherwise chunks go through the staging area.
    double *drho = rho ? device_view(rho) : nullptr, *du = u ? device_view(u) : nullptr;
    double *dp = p ? device_view(p) : nullptr;
    if ((!rho || drho) && (!u || du) && (!p || dp)) {
        h->L->moments(h->kp, pops_ptr(h), psi_ptr(h), h->odd, drho, du, dp, 0, n, h->stream);
        int st = check_launch();
        if (st) return st;
        return plb_status(h);
    }
    double *stg = staging_ptr(h);
    for (long long c0 = 0; c0 < n; c0 += chunk) {
        const long long cn = (n - c0) < chunk ? (n - c0) : chunk;
        double *srho = stg, *su = stg + cn, *sp = stg + (1 + D) * cn;
        h->L->moments(h->kp, pops_ptr(h), psi_ptr(h), h->odd, rho ? srho : nullptr, u ? su : nullptr,
                      p ? sp : nullptr, c0, cn, h->stream);
        int st = check_launch();
        if (st) return st;
        if (rho) PLB_CUDA(cudaMemcpyAsync(rho + c0, srho, cn * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        if (u)
            for (int a = 0; a < D; ++a)
                PLB_CUDA(cudaMemcpyAsync(u + a * n + c0, su + a * cn, cn * sizeof(double), cudaMemcpyDeviceToHost,
                                         h->stream));
        if (p) PLB_CUDA(cudaMemcpyAsync(p + c0, sp, cn * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    }
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    return plb_status(h);
}

int plb_reduce(plb_t *h, int what, const int lo[3], const int hi[3], double *out) {
    if (!h || !out) return fail(PLB_EINVAL, "NULL argument");
    if (what < PLB_MASS || what > PLB_MEAN_P) return fail(PLB_EINVAL, "unknown reduction %d", what);
    int blo[3] = {0, 0, 0}, bhi[3] = {h->dims[0], h->dims[1], h->dims[2]};
    if (lo)
        for (int a = 0; a < 3; ++a) blo[a] = lo[a] < 0 ? 0 : lo[a];
    if (hi)
        for (int a = 0; a < 3; ++a) bhi[a] = hi[a] > h->dims[a] ? h->dims[a] : hi[a];
    long long count = 1;
    for (int a = 0; a < 3; ++a) count *= (bhi[a] > blo[a] ? bhi[a] - blo[a] : 0);
    if (count == 0) return fail(PLB_EINVAL, "empty box");
    const bool needs_force = what == PLB_MOMENTUM || what == PLB_UMAX || what == PLB_UL1 || what == PLB_UL2;
    if (needs_force) h->L->psi(h->kp, pops_ptr(h), psi_ptr(h), h->odd, h->stream);
    long long nb = (h->lay.n + 255) / 256;
    const int nblocks = (int)(nb < h->lay.max_blocks ? nb : h->lay.max_blocks);
    double *partials = h->partials;
    double *dout = h->out;
    const bool whole = blo[0] == 0 && blo[1] == 0 && blo[2] == 0 && bhi[0] == h->dims[0] &&
                       bhi[1] == h->dims[1] && bhi[2] == h->dims[2];
    if (what == PLB_MASS && whole)
        h->L->mass(h->kp, pops_ptr(h), partials, nblocks, h->stream);
    else
        h->L->reduce(h->kp, pops_ptr(h), psi_ptr(h), h->odd, what, blo, bhi, partials, nblocks, h->stream);
    int st = check_launch();
    if (st) return st;
    reduce_final_launch(partials, nblocks, what == PLB_UMAX, h->kp.flags, dout, h->stream);
    st = check_launch();
    if (st) return st;
    double res[plb::kReduceOut];
    PLB_CUDA(cudaMemcpyAsync(res, dout, sizeof(res), cudaMemcpyDeviceToHost, h->stream));
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    switch (what) {
        case PLB_MOMENTUM: out[0] = res[0]; out[1] = res[1]; out[2] = res[2]; break;
        case PLB_UL2: out[0] = std::sqrt(res[0]); break;
        case PLB_MEAN_RHO:
        case PLB_MEAN_P: out[0] = res[0] / (double)count; break;
        default: out[0] = res[0];
    }
    return status_of((unsigned)res[4]);
}

int plb_get_populations(plb_t *h, double *f) {
    if (!h || !f) return fail(PLB_EINVAL, "NULL argument");
    const long long n = h->lay.n, chunk = h->lay.chunk;
    double *stg = staging_ptr(h);
    for (long long c0 = 0; c0 < n; c0 += chunk) {
        const long long cn = (n - c0) < chunk ? (n - c0) : chunk;
        h->L->get_pops(h->kp, pops_ptr(h), h->odd, stg, c0, cn, h->stream);
        int st = check_launch();
        if (st) return st;
        for (int i = 0; i < h->lay.Q; ++i)
            PLB_CUDA(cudaMemcpyAsync(f + i * n + c0, stg + i * cn, cn * sizeof(double), cudaMemcpyDeviceToHost,
                                     h->stream));
    }
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    return PLB_OK;
}

int plb_set_populations(plb_t *h, const double *f) {
    if (!h || !f) return fail(PLB_EINVAL, "NULL argument");
    if (h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: populations are read-only here");
    const long long n = h->lay.n, chunk = h->lay.chunk;
    double *stg = staging_ptr(h);
    PLB_CUDA(forget_timeout(h));
    for (long long c0 = 0; c0 < n; c0 += chunk) {
        const long long cn = (n - c0) < chunk ? (n - c0) : chunk;
        for (int i = 0; i < h->lay.Q; ++i)
            PLB_CUDA(cudaMemcpyAsync(stg + i * cn, f + i * n + c0, cn * sizeof(double), cudaMemcpyHostToDevice,
                                     h->stream));
        h->L->set_pops(h->kp, pops_ptr(h), stg, c0, cn, h->stream);
        int st = check_launch();
        if (st) return st;
    }
    h->odd = 0;
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    return PLB_OK;
}

size_t plb_state_bytes(const plb_t *h) {
    if (!h) return 0;
    return 64 + (size_t)h->lay.Q * h->lay.pstride * h->lay.s_pop;
}

int plb_get_state(plb_t *h, void *host_buf, size_t bytes) {
    if (!h || !host_buf) return fail(PLB_EINVAL, "NULL argument");
    if (bytes < plb_state_bytes(h)) return fail(PLB_ENOMEM, "state buffer too small");
    long long hdr[8] = {(long long)MAGIC, h->lattice, h->opts.precision, h->dims[0], h->dims[1], h->dims[2], h->t,
                        h->odd};
    std::memcpy(host_buf, hdr, sizeof(hdr));
    PLB_CUDA(cudaMemcpyAsync(static_cast<char *>(host_buf) + 64, pops_ptr(h), plb_state_bytes(h) - 64,
                             cudaMemcpyDeviceToHost, h->stream));
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    return PLB_OK;
}

int plb_set_state(plb_t *h, const void *host_buf, size_t bytes) {
    if (!h || !host_buf) return fail(PLB_EINVAL, "NULL argument");
    if (h->view) return fail(PLB_EINVAL, "this lattice belongs to a batch: its state is read-only here");
    if (bytes < plb_state_bytes(h)) return fail(PLB_ENOMEM, "state buffer too small");
    long long hdr[8];
    std::memcpy(hdr, host_buf, sizeof(hdr));
    if (hdr[0] != (long long)MAGIC || hdr[1] != h->lattice || hdr[2] != h->opts.precision || hdr[3] != h->dims[0] ||
        hdr[4] != h->dims[1] || hdr[5] != h->dims[2])
        return fail(PLB_EINVAL, "state does not match this lattice");
    PLB_CUDA(forget_timeout(h));
    PLB_CUDA(cudaMemcpyAsync(pops_ptr(h), static_cast<const char *>(host_buf) + 64, plb_state_bytes(h) - 64,
                             cudaMemcpyHostToDevice, h->stream));
    PLB_CUDA(cudaStreamSynchronize(h->stream));
    h->t = hdr[6];
    h->odd = (int)hdr[7];
    return PLB_OK;
}

}  // extern "C"

// Final pass of the reductions: one warp per component sums every 32nd block's partial in each lane,
// then the lanes, in a fixed order (one thread adding all 1024 in turn is a 30 us chain of FP64
// additions).  The lattice's error flags ride along in out[4].
namespace {
__global__ void k_reduce_final(const double *__restrict__ partials, int nblocks, int is_max,
                               const unsigned *__restrict__ flags, double *__restrict__ out) {
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = 0.0;
    for (int b = lane; b < nblocks; b += 32) v = is_max ? fmax(v, partials[b * 4 + c]) : v + partials[b * 4 + c];
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_down_sync(0xffffffffu, v, o);
        v = is_max ? fmax(v, w) : v + w;
    }
    if (lane == 0) out[c] = v;
    if (threadIdx.x == 0) out[4] = (double)*flags;
}

void reduce_final_launch(const double *partials, int nblocks, int is_max, const unsigned *flags, double *out,
                         cudaStream_t st) {
    k_reduce_final<<<1, 128, 0, st>>>(partials, nblocks, is_max, flags, out);
}
}  // namespace
