// Internal declarations shared by the host code (C++) and the kernels (CUDA).
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/dg.h"
#include "dg_device.h"

namespace dg {

// Host-built reference data (FP64): quadrature, basis tables and the face
// point permutations for the 6 relative orientations.
struct RefData {
    int p = 0;
    std::vector<double> vol_xi;    // [Nq][3] reference coordinates
    std::vector<double> vol_w;     // [Nq]
    std::vector<double> face_bary; // [Nqf][3] barycentrics on the face's 3 vertices
    std::vector<double> face_w;    // [Nqf]
    std::vector<double> tab;       // TabLayout(p).total values
    std::vector<int8_t> fperm;     // [6][Nqf]
};

bool build_reference(int p, RefData& out, std::string& err);
void eval_basis(int p, const double xi[3], double* phi, double* grad /* [Nb][3] or null */);
extern const int kPerm3[6][3];     // the 6 permutations of (0,1,2), indexed by orientation code

// Face code of an interior (element, local face): bits 0-1 the neighbour's
// local face, bits 2-4 the orientation code.  Boundary faces store the
// negative neighbour id -1 - bc_type instead.
struct MeshHost {
    int64_t ne = 0, n_faces = 0, n_bfaces = 0, bw_before = 0, bw_after = 0;
    std::vector<int32_t> perm;     // perm[internal] = caller index
    std::vector<int32_t> iperm;    // iperm[caller] = internal index
    std::vector<int32_t> nbr;      // [ne][4] internal order
    std::vector<uint8_t> fcode;    // [ne][4]
    std::vector<double> jinv;      // [ne][9] internal order, row-major J^-1
    std::vector<double> x0J;       // [ne][12] caller order: x0 (3) then J row-major (9)
};

bool build_mesh(const int32_t* tet_vid, const double* tet_xyz, const int8_t* bc_tag, int64_t ne,
                int renumber, MeshHost& out, int& code, std::string& err);

// A face that a mesh evaluates, from one of its slots 4 e + f (on its owner's side, unless the owner
// is a halo element of a partition).  A boundary face belongs to its element; an interior face to the element
// with the smaller caller index, so the choice, like every other input of the face flux, does not
// depend on the internal element order.
struct FaceRec {
    int32_t slot;
    int32_t other;      // the matching slot, or -1 - bc_type
    int32_t code;       // bits 0-2 the orientation (face-point permutation), bit 3 set if slot owns the face
    int32_t owner;      // the owning slot in the numbers of the whole mesh
};

}  // namespace dg

struct dg_mesh {
    int p = 1, nb = 4, nq = 4, nqf = 3;
    int precision = DG_FP64, flux = DG_RUSANOV;
    double gamma = 1.4, roe_eps = 0.0, finf[5] = {0, 0, 0, 0, 0};
    int device = 0;
    bool has_bc = false, has_state = false;
    dg::MeshHost host;
    dg::RefData ref;
    // device buffers
    int32_t* d_nbr = nullptr;
    int32_t* d_bface = nullptr;    // boundary (element, face) codes 4 e + f, ascending (internal order)
    uint8_t* d_fcode = nullptr;
    int32_t* d_perm = nullptr;     // internal -> caller
    void* d_jinv = nullptr;        // Real [ne][9]
    double* d_jinv64 = nullptr;    // FP64 copy for reductions
    void* d_tab = nullptr;         // Real tables
    double* d_tab64 = nullptr;     // FP64 tables (projection, integrals)
    int8_t* d_fperm = nullptr;
    uint16_t* d_tab16 = nullptr;   // f16 operand images of the tables (mixed precision)
    float mix_inv_b1 = 1.f, mix_inv_b2 = 1.f;
    // mixed precision: per tile of consecutive elements, the slot codes, the cross and work
    // lists and the tile headers (build_mixed_tiles)
    uint32_t* d_mslot = nullptr;
    uint8_t* d_mlist = nullptr;
    int32_t* d_mhdr = nullptr;
    int32_t* d_mxnbr = nullptr;
    void* d_B[3] = {nullptr, nullptr, nullptr};   // state buffers (internal precision)
    // adjoint work buffers, one allocation d_adj (lazy): states d_V, and the face buffers below
    void* d_adj = nullptr;
    void* d_V[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    // residual / totals work buffers (lazy): a caller's state in internal order, and the residual
    // in internal order; kept apart from d_B so these calls never touch an RK step in progress
    void* d_W[2] = {nullptr, nullptr};
    double* d_io = nullptr;        // FP64 [ne][5][Nb] staging for host copies
    double* d_red = nullptr;       // reduction scratch
    double* h_red = nullptr;       // pinned host reduction result
    unsigned int* d_status = nullptr;
    // Navier-Stokes, one allocation (lazy): auxiliary gradient [ne][3][5][Nb], own viscous face fluxes
    // [ne][4][4][Nqf] and, in FP32 where there is room, traces of U [ne][4][5][Nqf] (FP64: d_T)
    double* d_Z = nullptr;
    double* d_HB = nullptr;
    void* d_TN = nullptr;
    // mixed precision, conservative mode-0 update (dg_set_conservative): per (element, face) flux
    // integrals [ne][4][5]; per slot the weight phi_0 2|S_f| / |det J| of the mode-0 pass and the
    // face's 2|S_f| (one value per face, in both slots)
    bool conservative = false;
    float* d_hs = nullptr;
    double* d_wslot = nullptr;
    double* d_farea = nullptr;
    // one evaluation per face (FP64, FP32): the faces this mesh evaluates (boundary faces last) with
    // their owners' outward normals, the number of elements with traces (own + halo on a
    // partition's mesh), and the face buffers [n_trace][4][5][Nqf] (traces, then the fluxes in their
    // place): d_T of the RK steps (FP64: of every residual; FP32: where the stages use it and there is
    // room); lazy, the adjoint's own: d_TA, d_TL the direction's traces
    bool face_once = false;
    dg::FaceRec* d_frec = nullptr;   // the allocation that holds the next two as well
    void* d_fnorm = nullptr;       // Real [n_flist][3]
    void* d_fscale = nullptr;      // Real [n_flist][2], the two sides' |grad lambda| (the adjoint)
    int64_t n_flist = 0, n_interior = 0, n_trace = 0;   // listed faces, interior ones among them
    void* d_T = nullptr;
    void *d_TA = nullptr, *d_TL = nullptr;
    bool faces_asked = false;      // d_T has been asked for after the creation
    size_t face_bytes() const;
    // small meshes: a CUDA graph of several captured RK3 steps at one dt (dg_rk3_step)
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t rk_exec = nullptr;
    double rk_graph_dt = -1.0;
    size_t state_bytes() const;
};

// Launchers (kernels.cu).  All return a cudaError_t of the launch.
namespace dg {
// T: the face buffer to use (null: the FP32 kernel that needs none)
cudaError_t launch_residual(dg_mesh* m, const void* U, const void* U0, void* out, int mode,
                            double dt, double a, double b, void* T, cudaStream_t s);
// the face-once path's device data for m, whose elements are [first, first + ne) of whole (m itself, or a
// partition's mesh in local numbers, own elements and then halo): the face list, boundary faces last,
// the owners' normals and, where the adjoint may want them, the two sides' scales, in one allocation; n_trace is the
// number of elements with traces
cudaError_t setup_face_once(dg_mesh* m, const dg_mesh* whole, int64_t first, int64_t n_trace, bool scales, cudaStream_t s);
size_t face_list_bytes(int64_t n, int precision, bool scales);
// face traces of two states of the mesh's precision (U1 may be null), into the face buffers T and T1
cudaError_t launch_traces2(dg_mesh* m, const void* U, void* T, const void* U1, void* T1, cudaStream_t s);
cudaError_t launch_gather(dg_mesh* m, const double* user, void* internal, cudaStream_t s);   // caller -> internal
cudaError_t launch_gather2(dg_mesh* m, const double* user, void* internal, const double* user1, void* internal1,
                           cudaStream_t s);   // two at once
cudaError_t launch_gather_f32(dg_mesh* m, const double* user, float* internal, cudaStream_t s);   // FP32 (a hi plane) only
// Navier-Stokes lines: the BR1 gradient into Z, then the viscous volume and face terms added to
// the residual R (internal order), in the mesh's arithmetic (FP64 meshes FP64; FP32 and mixed
// meshes FP32, U the state's hi plane); per element of that type T holds 20 Nqf values (the traces
// of U; null for the passes that need none, which the mixed forms always take), Z 15 Nb and HB
// ns_face_buffer_values
cudaError_t launch_ns_viscous(dg_mesh* m, const void* U, void* T, void* Z, void* HB, void* R, double mu, double prandtl,
                              cudaStream_t s);
// in FP32 without a trace buffer (mixed and FP32 meshes)
cudaError_t launch_ns_viscous_mixed(dg_mesh* m, const float* U, float* Z, float* HB, float* R, double mu, double prandtl,
                                    cudaStream_t s);
size_t ns_face_buffer_values(int p, int64_t ne);
// SSP-RK3 stage from a stored residual, out = a U0 + b (U + dt R), in the mesh's state format (the
// mixed forms: float-float planes, FP32 residual)
cudaError_t launch_rk_axpy(dg_mesh* m, const void* U, const void* U0, const void* R, void* out, double dt, double a,
                           double b, cudaStream_t s);
cudaError_t launch_scatter(dg_mesh* m, const void* internal, double* user, cudaStream_t s);  // internal -> caller
cudaError_t launch_scatter_f32(dg_mesh* m, const float* internal, double* user, cudaStream_t s);
cudaError_t launch_stable_dt(dg_mesh* m, const void* U, double* d_out, cudaStream_t s);
cudaError_t launch_integrals(dg_mesh* m, const void* U, double* d_out6, cudaStream_t s);
cudaError_t launch_boundary_flux(dg_mesh* m, const void* U, double* d_partial, double* d_out5, cudaStream_t s);
cudaError_t launch_applied_boundary_flux(dg_mesh* m, double* d_partial, double* d_out5, cudaStream_t s);
cudaError_t launch_project(dg_mesh* m, const double* f, double* U, cudaStream_t s);
cudaError_t launch_volume_points(dg_mesh* m, const double* d_x0J, double* xyz, cudaStream_t s);
cudaError_t launch_residual_vjp(dg_mesh* m, const void* U, const void* lam, const void* X, const void* Y,
                                const void* Z, const double c[4], void* out, cudaStream_t s);
cudaError_t launch_ke_grad(dg_mesh* m, const double* U_user, double* out_user, cudaStream_t s);
// mixed precision (tensor cores): state stored as float-float planes (hi, then lo)
cudaError_t launch_residual_mixed(dg_mesh* m, const float* U_hi, const float* U_lo, const float* U0_hi,
                                  const float* U0_lo, float* out_hi, float* out_lo, int mode, double dt, double a,
                                  double b, cudaStream_t s);
void build_mixed_tables(int p, bool bf16, const RefData& ref, std::vector<uint16_t>& out, float& inv_b1,
                        float& inv_b2);
void build_mixed_tiles(const MeshHost& h, std::vector<uint32_t>& slot, std::vector<uint8_t>& lists,
                       std::vector<int32_t>& hdr, std::vector<int32_t>& xnbr);
dg_status set_error(dg_status code, const char* msg);   // sets dg_last_error() for the calling thread
int mixed_tab_halves(int p);
}  // namespace dg
