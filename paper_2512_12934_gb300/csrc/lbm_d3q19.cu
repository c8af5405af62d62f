// D3Q19 two-component MRT pseudopotential step with the corrected open faces
// (the three-dimensional counterpart of lbm_d2q9.cu).
//
// One time step is five launches (plain, or replayed from graphs in two
// branches: launch_step_forked):
//   A  d3q_pull_kernel      pull streaming (Eq. 2) with halfway bounce-back
//                           (Eq. B1) and periodic wrap (Eq. B2) of interior
//                           nodes; component densities rho_k (= psi_k) to a
//                           field.
//   A' d3q_face_pull_kernel one thread per open-face slot: the same pull,
//                           then inlet reconstruction (Eq. 13 over the 5
//                           unknowns, alpha correction Eqs. 15-19) or the
//                           convective outlet (Eq. 20); densities.
//   B  d3q_collide_kernel   (FP32: d3q_collide_f32_kernel) rho of a 32x4x2 tile
//                           plus a 2-node halo (ghost mirrors of Eqs. 24-25) staged
//                           in shared memory; forces of Eqs. 10-11 on the
//                           92-vector 8th-order isotropic stencil; common
//                           velocity (Eqs. 7-8); MRT collision with forcing
//                           (Eqs. 1, 3-6, 9) with the 19x19 transforms
//                           unrolled over compile-time constants; per-face-node
//                           FP64 flux terms.
//   B' d3q_outlet_kernel    outlet nodes: normal velocity chi times that of the
//                           inward neighbour (Eq. 22), collision.
//   C  d3q_reduce_kernel    fixed-order FP64 sums of the flux terms: lambda
//                           (Eq. 21) and chi (Eq. 23) for the next step.
// Face nodes carry their post-boundary populations from A' to B, the outlet's
// previous post-boundary populations (Eq. 20) and the forces the inlet needs
// one step later in small slot-indexed arrays.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "lbm_d3q19.h"

namespace lbm3 {

// ---- lattice (velocity order: rest, +-x, +-y, +-z, the xy, xz, yz edges) ----
__host__ __device__ constexpr int ex_(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1
                                                                 : 0;
}
__host__ __device__ constexpr int ey_(int i) {
    return (i == 3 || i == 7 || i == 8 || i == 15 || i == 17) ? 1
           : (i == 4 || i == 9 || i == 10 || i == 16 || i == 18) ? -1
                                                                 : 0;
}
__host__ __device__ constexpr int ez_(int i) {
    return (i == 5 || i == 11 || i == 12 || i == 15 || i == 16) ? 1
           : (i == 6 || i == 13 || i == 14 || i == 17 || i == 18) ? -1
                                                                  : 0;
}
__host__ __device__ constexpr int e2_(int i) { return ex_(i) * ex_(i) + ey_(i) * ey_(i) + ez_(i) * ez_(i); }
__host__ __device__ constexpr int opp_(int i) {
    for (int j = 0; j < Q; ++j)
        if (ex_(j) == -ex_(i) && ey_(j) == -ey_(i) && ez_(j) == -ez_(i)) return j;
    return 0;
}
// weights times 36
__host__ __device__ constexpr int w36_(int i) { return e2_(i) == 0 ? 12 : (e2_(i) == 1 ? 2 : 1); }

// Orthogonal moment basis: rho, e, eps, j_x, q_x, j_y, q_y, j_z, q_z, 3p_xx,
// 3pi_xx, p_ww, pi_ww, p_xy, p_yz, p_xz, m_x, m_y, m_z.
__host__ __device__ constexpr int T_(int r, int i) {
    const int x = ex_(i), y = ey_(i), z = ez_(i), e2 = e2_(i);
    switch (r) {
    case 0: return 1;
    case 1: return 19 * e2 - 30;
    case 2: return (21 * e2 * e2 - 53 * e2 + 24) / 2;
    case 3: return x;
    case 4: return (5 * e2 - 9) * x;
    case 5: return y;
    case 6: return (5 * e2 - 9) * y;
    case 7: return z;
    case 8: return (5 * e2 - 9) * z;
    case 9: return 3 * x * x - e2;
    case 10: return (3 * e2 - 5) * (3 * x * x - e2);
    case 11: return y * y - z * z;
    case 12: return (3 * e2 - 5) * (y * y - z * z);
    case 13: return x * y;
    case 14: return y * z;
    case 15: return x * z;
    case 16: return (y * y - z * z) * x;
    case 17: return (z * z - x * x) * y;
    default: return (x * x - y * y) * z;
    }
}
__host__ __device__ constexpr int Tnorm_(int r) {
    int s = 0;
    for (int i = 0; i < Q; ++i) s += T_(r, i) * T_(r, i);
    return s;
}

// 8th-order isotropic stencil weights (second moment 1) by |e|^2, times 5040
__host__ __device__ constexpr int sw5040_(int r2) {
    return r2 == 1 ? 448 : r2 == 2 ? 240 : r2 == 3 ? 96 : r2 == 4 ? 50 : r2 == 5 ? 16 : r2 == 6 ? 8 : r2 == 8 ? 1 : 0;
}

// Compile-time loop: f(std::integral_constant<int, i>) for i in [B, E), so
// every lattice constant below is a template constant (no runtime tables).
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (B < E) {
        f(std::integral_constant<int, B>{});
        static_for<B + 1, E>(f);
    }
}

// acc += c * v with the integer c folded at compile time (0: nothing).
template <int c, typename R>
__device__ __forceinline__ void acc_c(R& acc, R v) {
    if constexpr (c == 1) acc += v;
    else if constexpr (c == -1) acc -= v;
    else if constexpr (c != 0) acc += (R)c * v;
}

// ---- tiles of the collide kernel -----------------------------------------
// Tiles are TX x TY x TZ nodes of one thread each.
constexpr int TX = 32, TY = 4;
constexpr int HX = TX + 4, HY = TY + 4;
template <typename S>
struct Tile3 {
    static constexpr int TZ = 2;
    static constexpr int HZ = TZ + 4;
    static constexpr int HN = HX * HY * HZ;
    static constexpr int NT = TX * TY * TZ;
    static constexpr int MIN_BLOCKS = sizeof(S) == 8 ? 1 : 3;
};
static_assert(HX == RHO_BOX3_X && HY == RHO_BOX3_Y && Tile3<float>::HZ == RHO_BOX3_Z,
              "the density tensor-copy box must be the FP32 collide tile plus its halo");

template <typename R>
struct Pair;
template <>
struct Pair<float> {
    using type = float2;
};
template <>
struct Pair<double> {
    using type = double2;
};

template <typename S>
struct Store;
template <>
struct Store<float> {
    using R = float;
};
template <>
struct Store<double> {
    using R = double;
};
template <>
struct Store<__half> {
    using R = float;
};

template <typename S>
__device__ __forceinline__ constexpr bool is_half() {
    return std::is_same<S, __half>::value;
}

// A stored population as a real number (FP16 storage: the deviation only).
template <typename S>
__device__ __forceinline__ typename Store<S>::R ld_pop(S v) {
    if constexpr (is_half<S>()) return __half2float(v);
    else return v;
}

// Density rounded to the half-precision reference of FP16 storage.
__device__ __forceinline__ float half_round(float r) { return __half2float(__float2half_rn(r)); }

// Wrap a pull source on periodic axes (blocked sources never reach here).
__device__ __forceinline__ int wrap(int c, int n) { return c < 0 ? c + n : (c >= n ? c - n : c); }

template <typename S>
__device__ __forceinline__ long long node_index(const D3Args<S>& a, int x, int y, int z) {
    return ((long long)z * a.ny + y) * a.pitch + x;
}

template <typename S>
__device__ __forceinline__ void st_at(S* base, unsigned off, S v) {
    *reinterpret_cast<S*>(reinterpret_cast<char*>(base) + off) = v;
}

// The pull sources of components [K0, K1) of node n = (x, y, z) (Eq. 2, Eq. B1,
// Eq. B2) as addresses: use(k, i, p).  Most nodes have no blocked direction and
// no wrap: the shifted planes.  The others select each source (its neighbour
// with periodic wraps, or the opposite direction of the node itself) without a
// branch, so that their loads are in flight together too: a branch per
// direction made every load wait for the one before it.  The offsets are
// 32-bit: n * 8 bytes stays below 2^32 for every grid that fits the device.
template <int K0, int K1, typename S, typename Use>
__device__ __forceinline__ void pull_sources(const D3Args<S>& a, int x, int y, int z, long long n, uint32_t info,
                                             Use use) {
    auto at = [](const S* base, unsigned m) {
        return reinterpret_cast<const S*>(reinterpret_cast<const char*>(base) + m * (unsigned)sizeof(S));
    };
    if ((info & (0x7FFFFu | INFO3_WRAP)) == 0u) {
        static_for<K0, K1>([&](auto K) {
            constexpr int k = decltype(K)::value;
            static_for<0, Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                use(k, i, at(a.src[k][i], (unsigned)n));
            });
        });
        return;
    }
    // index distances to the (wrapped) neighbours; that of a blocked source is not used
    const int sz = a.ny * a.pitch;
    const int dxm = wrap(x - 1, a.nx) - x, dxp = wrap(x + 1, a.nx) - x;
    const int dym = (wrap(y - 1, a.ny) - y) * a.pitch, dyp = (wrap(y + 1, a.ny) - y) * a.pitch;
    const int dzm = (wrap(z - 1, a.nz) - z) * sz, dzp = (wrap(z + 1, a.nz) - z) * sz;
    static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        const bool bb = (info & (1u << i)) != 0;
        const int d = (ex_(i) == 1 ? dxm : (ex_(i) == -1 ? dxp : 0)) + (ey_(i) == 1 ? dym : (ey_(i) == -1 ? dyp : 0)) +
                      (ez_(i) == 1 ? dzm : (ez_(i) == -1 ? dzp : 0));
        const unsigned m = (unsigned)n + (unsigned)(bb ? 0 : d);
        static_for<K0, K1>([&](auto K) {
            constexpr int k = decltype(K)::value;
            use(k, i, at(a.fin + (bb ? k * Q + opp_(i) : k * Q + i) * a.plane, m));
        });
    });
}

// Raw pull of component K at node n.
template <int K, typename S>
__device__ __forceinline__ void pull_raw(const D3Args<S>& a, int x, int y, int z, long long n, uint32_t info,
                                         S (&v)[Q]) {
    pull_sources<K, K + 1>(a, x, y, z, n, info, [&](int, int i, const S* p) { v[i] = __ldg(p); });
}

// Pull of component k as real values.
template <int k, typename S, typename R>
__device__ __forceinline__ void pull(const D3Args<S>& a, int x, int y, int z, uint32_t info, R (&f)[Q]) {
    const long long n = node_index(a, x, y, z);
    // FP16 storage: every value this node pulls was encoded against its
    // reference density (the writer used the same half-rounded density)
    R ref = 0;
    if constexpr (is_half<S>()) ref = __half2float(a.rref_in[(size_t)k * a.plane + n]);
    S v[Q];
    pull_raw<k>(a, x, y, z, n, info, v);
    static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        f[i] = (R)ld_pop(v[i]);
        if constexpr (is_half<S>()) f[i] += ((R)w36_(i) / (R)36) * ref;
    });
}

template <typename R>
__device__ __forceinline__ void feq(R rho, R ux, R uy, R uz, R (&out)[Q]) {
    const R uu = ux * ux + uy * uy + uz * uz;
    static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        R eu = 0;
        acc_c<ex_(i)>(eu, ux);
        acc_c<ey_(i)>(eu, uy);
        acc_c<ez_(i)>(eu, uz);
        out[i] = rho * ((R)w36_(i) / (R)36) * ((R)1 + (R)3 * eu + (R)4.5 * eu * eu - (R)1.5 * uu);
    });
}

// Density as the rest population plus the sums of opposite pairs.
template <typename R>
__device__ __forceinline__ R sum19(const R (&f)[Q]) {
    R s = f[0];
    static_for<1, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (opp_(i) > i) s += f[i] + f[opp_(i)];
    });
    return s;
}

// Momentum as sums of opposite-pair differences (each difference of two
// nearby populations is exact or nearly so, which keeps FP32 j accurate).
template <typename R>
__device__ __forceinline__ void moments_j(const R (&f)[Q], R& jx, R& jy, R& jz) {
    R x = 0, y = 0, z = 0;
    static_for<1, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (opp_(i) > i) {
            const R d = f[i] - f[opp_(i)];
            acc_c<ex_(i)>(x, d);
            acc_c<ey_(i)>(y, d);
            acc_c<ez_(i)>(z, d);
        }
    });
    jx = x;
    jy = y;
    jz = z;
}

// Eq. 1 for one component: f <- f - T^-1 S (T f - m^eq) + T^-1 (I - S/2) F_m,
// T^-1 = T^T diag(1/|row|^2) (orthogonal rows).  m^eq = T f^eq and F_m =
// T Fbar (Eqs. 6, 9) are written out as the polynomials they reduce to for
// this basis (rho; e: rho(19u^2 - 11); eps: rho(6 - 11u^2)/2; j: rho u;
// q: -2 rho u/3; 3p_xx: rho(3u_x^2 - u^2); 3pi_xx: -3p_xx/2; p_ww:
// rho(u_y^2 - u_z^2); pi_ww: -p_ww/2; p_ab: rho u_a u_b; m: 0 -- and for
// F_m the same moments of the Guo term: 0, 38 u.F, -11 u.F, F, -2F/3,
// 2(3u_xF_x - u.F), -(3u_xF_x - u.F), 2(u_yF_y - u_zF_z), -(u_yF_y - u_zF_z),
// u_aF_b + u_bF_a, 0).  All entries of T are template constants.
// Moments through opposite pairs: the even rows of T (rho, e, eps, p, pi)
// weigh f_i and f_ibar alike, the odd rows (j, q, m) with opposite signs, so
// T f needs only the pair sums P_i = f_i + f_ibar and differences
// D_i = f_i - f_ibar (i over one member of each pair), and the back
// transform splits the same way.
template <int r>
__host__ __device__ constexpr bool odd_row() {
    return r == 3 || r == 4 || r == 5 || r == 6 || r == 7 || r == 8 || r == 16 || r == 17 || r == 18;
}

template <typename R>
__device__ __forceinline__ void collide(R (&f)[Q], R rho, R ux, R uy, R uz, R Fx, R Fy, R Fz, const R* s) {
    R P[Q], D[Q];  // only the entries of the first member of each pair are used
    static_for<1, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (opp_(i) > i) {
            P[i] = f[i] + f[opp_(i)];
            D[i] = f[i] - f[opp_(i)];
        }
    });
    R m[Q];
    static_for<0, Q>([&](auto Rr) {
        constexpr int r = decltype(Rr)::value;
        R acc = 0;
        if constexpr (!odd_row<r>()) acc_c<T_(r, 0)>(acc, f[0]);
        static_for<1, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if constexpr (opp_(i) > i) {
                if constexpr (odd_row<r>()) acc_c<T_(r, i)>(acc, D[i]);
                else acc_c<T_(r, i)>(acc, P[i]);
            }
        });
        m[r] = acc;
    });
    const R uu = ux * ux + uy * uy + uz * uz;
    const R uF = ux * Fx + uy * Fy + uz * Fz;
    const R pxx = (R)2 * ux * ux - uy * uy - uz * uz, fxx = (R)2 * ((R)2 * ux * Fx - uy * Fy - uz * Fz);
    const R pww = uy * uy - uz * uz, fww = (R)2 * (uy * Fy - uz * Fz);
    const R meq[Q] = {rho, rho * ((R)19 * uu - (R)11), rho * ((R)6 - (R)11 * uu) * (R)0.5, rho * ux,
                      -(R)2 / (R)3 * rho * ux, rho * uy, -(R)2 / (R)3 * rho * uy, rho * uz, -(R)2 / (R)3 * rho * uz,
                      rho * pxx, -(R)0.5 * rho * pxx, rho * pww, -(R)0.5 * rho * pww, rho * ux * uy, rho * uy * uz,
                      rho * ux * uz, 0, 0, 0};
    const R mF[Q] = {0, (R)38 * uF, -(R)11 * uF, Fx, -(R)2 / (R)3 * Fx, Fy, -(R)2 / (R)3 * Fy, Fz,
                     -(R)2 / (R)3 * Fz, fxx, -(R)0.5 * fxx, fww, -(R)0.5 * fww, ux * Fy + uy * Fx, uy * Fz + uz * Fy,
                     ux * Fz + uz * Fx, 0, 0, 0};
    R g[Q];
    static_for<0, Q>([&](auto Rr) {
        constexpr int r = decltype(Rr)::value;
        // the density row drops out: m_rho = m^eq_rho by definition and the
        // forcing term has no density moment
        if constexpr (r == 0) g[r] = (R)0;
        else g[r] = (-s[r] * (m[r] - meq[r]) + ((R)1 - (R)0.5 * s[r]) * mF[r]) * ((R)1 / (R)Tnorm_(r));
    });
    {
        R acc = 0;
        static_for<0, Q>([&](auto Rr) {
            constexpr int r = decltype(Rr)::value;
            acc_c<T_(r, 0)>(acc, g[r]);
        });
        f[0] += acc;
    }
    static_for<1, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (opp_(i) > i) {
            R ev = 0, od = 0;
            static_for<0, Q>([&](auto Rr) {
                constexpr int r = decltype(Rr)::value;
                if constexpr (odd_row<r>()) acc_c<T_(r, i)>(od, g[r]);
                else acc_c<T_(r, i)>(ev, g[r]);
            });
            f[i] += ev + od;
            f[opp_(i)] += ev - od;
        }
    });
}

// ---- kernel A: pull, open faces, densities --------------------------------
template <typename S>
__device__ void face_reconstruct(const D3Args<S>& a, int fid, int x, int y, int z, uint32_t info,
                                 typename Store<S>::R (&f)[2][Q]) {
    using R = typename Store<S>::R;
    const FaceDev3& F = a.face[fid];
    const int ox = F.o[0], oy = F.o[1], oz = F.o[2];
    const int slot = face_slot(F, x, y, z);
    const int x2 = x - ox, y2 = y - oy, z2 = z - oz;
    const uint32_t info2 = a.info[node_index(a, x2, y2, z2)];
    if (F.kind == FACE3_INLET) {
        R f2[2][Q];
        pull<0, S, R>(a, x2, y2, z2, info2, f2[0]);
        pull<1, S, R>(a, x2, y2, z2, info2, f2[1]);
        const R* Fp2 = a.FpN + (size_t)slot * 6;
        const R* Fp1 = a.FpF + (size_t)slot * 6;
        R r2[2], jx = 0, jy = 0, jz = 0;
        #pragma unroll
        for (int k = 0; k < 2; ++k) {
            r2[k] = sum19(f2[k]);
            R x_, y_, z_;
            moments_j(f2[k], x_, y_, z_);
            jx += x_ + (R)0.5 * Fp2[k * 3 + 0];
            jy += y_ + (R)0.5 * Fp2[k * 3 + 1];
            jz += z_ + (R)0.5 * Fp2[k * 3 + 2];
        }
        const R rt2 = r2[0] + r2[1];
        const R u2x = jx / rt2, u2y = jy / rt2, u2z = jz / rt2;
        const R speed = (R)a.face_speed[slot];
        const R uin[3] = {-(R)ox * speed, -(R)oy * speed, -(R)oz * speed};
        #pragma unroll
        for (int k = 0; k < 2; ++k) {
            const R rin = (R)a.face_rho[(size_t)k * a.nface_slots + slot];
            R e1[Q], e2[Q];
            feq(rin, uin[0], uin[1], uin[2], e1);
            feq(r2[k], u2x, u2y, u2z, e2);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (ex_(i) * ox + ey_(i) * oy + ez_(i) * oz < 0) f[k][i] = e1[i] + (f2[k][i] - e2[i]);
            if (F.alpha) {
                R mx, my, mz;
                moments_j(f[k], mx, my, mz);
                const R dx = rin * uin[0] - (mx + (R)0.5 * Fp1[k * 3 + 0]);
                const R dy = rin * uin[1] - (my + (R)0.5 * Fp1[k * 3 + 1]);
                const R dz = rin * uin[2] - (mz + (R)0.5 * Fp1[k * 3 + 2]);
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    if (ex_(i) * ox + ey_(i) * oy + ez_(i) * oz < 0)
                        f[k][i] += ((R)w36_(i) / (R)36) *
                                   ((R)ex_(i) * dx / (R)F.sa[0] + (R)ey_(i) * dy / (R)F.sa[1] +
                                    (R)ez_(i) * dz / (R)F.sa[2]);
            }
        }
    } else {
        // convective outlet (Eq. 20) with lambda of the previous step
        R fN1[2][Q];
        pull<0, S, R>(a, x2, y2, z2, info2, fN1[0]);
        pull<1, S, R>(a, x2, y2, z2, info2, fN1[1]);
        const R lam = (R)a.scal_in[SC3_LAMBDA];
        R* fo = a.fo + (size_t)slot * 2 * Q;
        #pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (ex_(i) * ox + ey_(i) * oy + ez_(i) * oz < 0)
                    f[k][i] = (fo[k * Q + i] + lam * fN1[k][i]) / ((R)1 + lam);
        }
        #pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int i = 0; i < Q; ++i) fo[k * Q + i] = f[k][i];
    }
    R* ff = a.fface + (size_t)slot * 2 * Q;
    #pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < Q; ++i) ff[k * Q + i] = f[k][i];
}

// One thread per node and component: the 19 loads of a thread fit 40 registers,
// so 48 warps an SM keep them in flight (both components in one thread, 24
// warps at 80 registers: 116 us on 512x96x96, this form 103; FP16 storage on
// 250x50x50: 18 us).
template <typename S>
__global__ void __launch_bounds__(256, sizeof(S) == 8 ? 3 : 6) d3q_pull_kernel(const __grid_constant__ D3Args<S> a, int zblock) {
    using R = typename Store<S>::R;
    const int x = blockIdx.x * 32 + threadIdx.x;
    const int y = blockIdx.y * 4 + threadIdx.y;
    const int z = zblock + blockIdx.z, k = threadIdx.z;
    if (x >= a.nx || y >= a.ny) return;
    const long long n = node_index(a, x, y, z);
    const uint32_t info = a.info[n];
    if ((info >> INFO3_FACE_SHIFT) & 7u) return;  // open-face nodes: d3q_face_pull_kernel
    R r = 0;                                      // psi = 0 at solid sites of the force stencil
    if (!(info & INFO3_SOLID)) {
        S v[Q];
        if (k == 0) pull_raw<0>(a, x, y, z, n, info, v);
        else pull_raw<1>(a, x, y, z, n, info, v);
        if constexpr (is_half<S>()) {
            // sum w_i = 1: rho_k = rho_ref + the sum of the stored deviations
            float acc = 0.0f;
            static_for<0, Q>([&](auto I) { acc += __half2float(v[decltype(I)::value]); });
            r = __half2float(a.rref_in[(size_t)k * a.plane + n]) + acc;
        } else {
            r = sum19(v);
        }
    }
    a.rho[2 * n + k] = r;
}

// Face slot -> face index and node coordinates; false for solid positions.
template <typename S>
__device__ __forceinline__ bool slot_node(const D3Args<S>& a, int slot, int& fid, int (&c)[3]) {
    if (slot >= a.nface_slots || !a.face_fluid[slot]) return false;
    fid = 0;
    while (fid + 1 < a.nfaces && slot >= a.face[fid + 1].base) ++fid;
    const FaceDev3& F = a.face[fid];
    const int q = slot - F.base;
    const int ext[3] = {a.nx, a.ny, a.nz};
    c[F.axis] = (F.side & 1) ? ext[F.axis] - 1 : 0;
    c[F.a0] = F.lo0 + q % F.len0;
    c[F.a1] = F.lo1 + q / F.len0;
    return true;
}

// One thread per face slot: pull, open-face reconstruction, densities.
template <typename S>
__global__ void __launch_bounds__(128) d3q_face_pull_kernel(D3Args<S> a) {
    using R = typename Store<S>::R;
    int fid, c[3];
    if (!slot_node(a, blockIdx.x * blockDim.x + threadIdx.x, fid, c)) return;
    const long long n = node_index(a, c[0], c[1], c[2]);
    const uint32_t info = a.info[n];
    R f[2][Q];
    pull<0, S, R>(a, c[0], c[1], c[2], info, f[0]);
    pull<1, S, R>(a, c[0], c[1], c[2], info, f[1]);
    face_reconstruct<S>(a, fid, c[0], c[1], c[2], info, f);
    reinterpret_cast<typename Pair<R>::type*>(a.rho)[n] = typename Pair<R>::type{sum19(f[0]), sum19(f[1])};
}

// ---- kernel B: forces, velocity, collision --------------------------------
// Resolve a psi / indicator site (Eqs. 10, 11, 24, 25) to a node index:
// periodic wrap, ghost mirror across open sides, -1 outside a closed side
// (a solid wall).  Solid nodes inside the grid carry (0, 0) in the density
// field: psi = 0 there, as at closed sides.
template <typename S>
__device__ __forceinline__ long long site_index(const D3Args<S>& a, int x, int y, int z) {
    int c[3] = {x, y, z};
    const int ext[3] = {a.nx, a.ny, a.nz};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (c[ax] >= 0 && c[ax] < ext[ax]) continue;
        if (a.periodic[ax]) c[ax] = c[ax] < 0 ? c[ax] + ext[ax] : c[ax] - ext[ax];
        else if (c[ax] < 0 && a.open_side[2 * ax]) c[ax] = -1 - c[ax];
        else if (c[ax] >= ext[ax] && a.open_side[2 * ax + 1]) c[ax] = 2 * ext[ax] - 1 - c[ax];
        else return -1;
    }
    return node_index(a, c[0], c[1], c[2]);
}

// Interaction sums over the 92-vector stencil: g_k = sum w psi_k(x+e) e,
// `site(dx, dy, dz)` returns the (psi_1, psi_2) pair of a site (0 at solids).
// Pairs (e, -e) share the weight: g += w e (psi(x+e) - psi(x-e)); c runs over
// the half of the 5x5x5 cube before its centre (index 62), -e is site 124 - c.
// In FP32 both components go through one packed FP32x2 operation per term
// (each lane rounds as the scalar FMA does).
template <typename R, typename Site>
__device__ __forceinline__ void stencil_sums(Site site, R (&g1)[3], R (&g2)[3]) {
    if constexpr (std::is_same<R, float>::value) {
        float2 g[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) g[q] = make_float2(0.f, 0.f);
        static_for<0, 62>([&](auto C) {
            constexpr int c = decltype(C)::value;
            constexpr int dx = c % 5 - 2, dy = (c / 5) % 5 - 2, dz = c / 25 - 2;
            constexpr int r2 = dx * dx + dy * dy + dz * dz;
            constexpr int wq = sw5040_(r2);
            if constexpr (wq != 0) {
                constexpr float w = (float)wq / 5040.f;
                const float2 d = __ffma2_rn(site(-dx, -dy, -dz), make_float2(-1.f, -1.f), site(dx, dy, dz));
                if constexpr (dx != 0) g[0] = __ffma2_rn(make_float2(w * dx, w * dx), d, g[0]);
                if constexpr (dy != 0) g[1] = __ffma2_rn(make_float2(w * dy, w * dy), d, g[1]);
                if constexpr (dz != 0) g[2] = __ffma2_rn(make_float2(w * dz, w * dz), d, g[2]);
            }
        });
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            g1[q] = g[q].x;
            g2[q] = g[q].y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) g1[q] = g2[q] = (R)0;
        static_for<0, 62>([&](auto C) {
            constexpr int c = decltype(C)::value;
            constexpr int dx = c % 5 - 2, dy = (c / 5) % 5 - 2, dz = c / 25 - 2;
            constexpr int r2 = dx * dx + dy * dy + dz * dz;
            constexpr int wq = sw5040_(r2);
            if constexpr (wq != 0) {
                const R w = (R)wq / (R)5040;
                const auto p = site(dx, dy, dz), m = site(-dx, -dy, -dz);
                const R d1 = p.x - m.x, d2 = p.y - m.y;
                if constexpr (dx != 0) {
                    g1[0] += (w * (R)dx) * d1;
                    g2[0] += (w * (R)dx) * d2;
                }
                if constexpr (dy != 0) {
                    g1[1] += (w * (R)dy) * d1;
                    g2[1] += (w * (R)dy) * d2;
                }
                if constexpr (dz != 0) {
                    g1[2] += (w * (R)dz) * d1;
                    g2[2] += (w * (R)dz) * d2;
                }
            }
        });
    }
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Wait for phase `parity` of an mbarrier for at most about a second of SM
// clock; false if the wait ran out.
__device__ __forceinline__ bool bar_wait(unsigned long long* bar, unsigned parity) {
    const long long t0 = clock64();
    for (;;) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(smem_addr(bar)), "r"(parity)
                     : "memory");
        if (done) return true;
        if (clock64() - t0 > 2000000000LL) return false;
    }
}

// The density box has landed.  If the wait runs out the status word says so, and
// the copy, which still writes this CTA's shared memory, is given as long again.
__device__ __forceinline__ void wait_box(unsigned long long* bar, unsigned* status, bool report) {
    if (bar_wait(bar, 0u)) return;
    if (report) atomicOr(status, STATUS3_TIMEOUT);
    bar_wait(bar, 0u);
}

__device__ __forceinline__ void bar_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// One tensor copy of the density box that starts at (x, y, z), `bytes` long,
// completing on phase 0 of `bar`.
__device__ __forceinline__ void copy_box(const CUtensorMap* map, void* dst, unsigned bytes, int x, int y, int z,
                                         unsigned long long* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
}

// sum_e w s(x+e) e of Eq. 11 (geometry only; precomputed per near-solid node)
template <typename S>
__device__ __forceinline__ void adhesion_vector(const D3Args<S>& a, long long n, uint32_t info,
                                                typename Store<S>::R (&ad)[3]) {
    using R = typename Store<S>::R;
    if (info & INFO3_NEAR_SOLID) {
        ad[0] = (R)a.adv[n];
        ad[1] = (R)a.adv[a.plane + n];
        ad[2] = (R)a.adv[2 * a.plane + n];
    } else {
        ad[0] = ad[1] = ad[2] = (R)0;
    }
}

template <typename R>
__device__ __forceinline__ void forces(const R* G, R r1, R r2, const R (&g1)[3], const R (&g2)[3], const R (&ad)[3],
                                       const R* body, R (&F1)[3], R (&F2)[3]) {
    // G = {G12, Gw1, Gw2}
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        F1[q] = -G[0] * r1 * g2[q] - G[1] * r1 * ad[q];
        F2[q] = -G[0] * r2 * g1[q] - G[2] * r2 * ad[q];
    }
    // six divisions that most runs (no body force) do without
    if (body[0] != (R)0 || body[1] != (R)0 || body[2] != (R)0) {
        const R rt = r1 + r2;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            F1[q] += body[q] * r1 / rt;
            F2[q] += body[q] * r2 / rt;
        }
    }
}

template <typename R>
__device__ __forceinline__ void add_j(const R (&f)[Q], R (&j)[3]) {
    R jx, jy, jz;
    moments_j(f, jx, jy, jz);
    j[0] += jx;
    j[1] += jy;
    j[2] += jz;
}

// Store the post-collision populations of component k at node n.  FP16
// storage writes half(f*_i - w_i rho_ref), rho_ref being the half-rounded
// density of component k at the node that pulls f*_i next step: x + e_i, or
// x itself when that neighbour is solid or outside (halfway bounce-back).
// dest_ref(I, k) returns that reference (already half-rounded).
template <typename S, typename DestRho>
__device__ __forceinline__ void store_pop(const D3Args<S>& a, int k, long long n, const typename Store<S>::R (&f)[Q],
                                          DestRho dest_ref) {
    using R = typename Store<S>::R;
    const unsigned off = (unsigned)n * (unsigned)sizeof(S);
    static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (is_half<S>()) {
            const R ref = dest_ref(I, k);
            st_at(a.dst[k][i], off, __float2half_rn(f[i] - ((R)w36_(i) / (R)36) * ref));
        } else {
            st_at(a.dst[k][i], off, (S)f[i]);
        }
    });
}

template <typename S>
__device__ __forceinline__ void check_store_u(const D3Args<S>& a, long long n, typename Store<S>::R rt,
                                              const typename Store<S>::R (&u)[3]) {
    if (!(isfinite((float)rt) && isfinite((float)u[0]) && isfinite((float)u[1]) && isfinite((float)u[2])))
        atomicOr(a.status, STATUS3_DIVERGED);
    if (a.umac) {
        a.umac[n] = u[0];
        a.umac[a.plane + n] = u[1];
        a.umac[2 * a.plane + n] = u[2];
    }
}

// Density box of a tile and its halo by loads: periodic wraps, ghost mirrors and
// walls resolved per site unless the whole box lies inside the grid.
template <typename S, typename Put>
__device__ __forceinline__ void stage_box(const D3Args<S>& a, int x0, int y0, int z0, bool inner, int tid, Put put) {
    using R = typename Store<S>::R;
    using V = typename Pair<R>::type;
    constexpr int HN = Tile3<S>::HN, NT = Tile3<S>::NT, PASSES = (HN + NT - 1) / NT;
    const V* rp = reinterpret_cast<const V*>(a.rho);
    V v[PASSES];
#pragma unroll
    for (int p = 0; p < PASSES; ++p) {  // every pass's load in flight before the first store
        const int q = p * NT + tid;
        v[p] = V{(R)0, (R)0};
        if (q < HN) {
            const int hx = q % HX, hy = (q / HX) % HY, hz = q / (HX * HY);
            const long long m = inner ? node_index(a, x0 - 2 + hx, y0 - 2 + hy, z0 - 2 + hz)
                                      : site_index(a, x0 - 2 + hx, y0 - 2 + hy, z0 - 2 + hz);
            if (m >= 0) v[p] = rp[m];
        }
    }
#pragma unroll
    for (int p = 0; p < PASSES; ++p)
        if (p * NT + tid < HN) put(p * NT + tid, v[p]);
}

// FP64 and FP16 storage.  Every fluid node of a 32x4x2 tile: forces from the
// staged densities (the halo resolves periodic wraps and the ghost mirrors of
// Eqs. 24-25), the common velocity, the collision of one component after the
// other.  Open-face nodes take their post-boundary populations from the face
// kernel; outlet nodes stop after the force (their normal velocity waits for
// the inward neighbour's, Eq. 22), and the inward neighbours of the outlet
// hand theirs over with the flux terms of Eqs. 21, 23.  Residency: FP16 storage
// 3 CTAs of 256 per SM (80 registers), FP64 1.  Tiles without a fluid node
// leave before staging.
template <typename S>
__global__ void __launch_bounds__(Tile3<S>::NT, Tile3<S>::MIN_BLOCKS)
    d3q_collide_kernel(const __grid_constant__ D3Args<S> a, const __grid_constant__ CUtensorMap rho_map, int use_tma,
                       int zblock) {
    using R = typename Store<S>::R;
    constexpr int TZ = Tile3<S>::TZ, HN = Tile3<S>::HN, NT = Tile3<S>::NT;
    __shared__ __align__(128) typename Pair<R>::type s_rr[HN];  // (rho_1, rho_2) of the tile and its halo
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ __half2 s_ref[is_half<S>() ? HN : 1];            // FP16 storage: the same rounded to half
    __shared__ R s_rate[2][Q];  // relaxation rates of both components (indexed by component below)
    // component 0's pulled populations, kept for its collision after
    // component 1's (FP16 storage; FP64 pulls them again, its tile would
    // exceed the static shared-memory limit)
    constexpr bool STASH = sizeof(R) == 4;
    __shared__ R s_f0[STASH ? Q : 1][STASH ? NT : 1];
    // from the last z on: the pull kernel has just read those planes (L2), and the
    // next one starts on the planes this kernel writes last (co-flow 250x64x64
    // 112.7 us per step in ascending order, 108.4 in this one; 512x96x96 400, 397)
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = (zblock + (int)(gridDim.z - 1 - blockIdx.z)) * TZ;
    const int tid = threadIdx.x + TX * (threadIdx.y + TY * threadIdx.z);
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    const bool in_grid = x < a.nx && y < a.ny && z < a.nz;
    const long long n = in_grid ? node_index(a, x, y, z) : 0;
    const uint32_t info = in_grid ? a.info[n] : (uint32_t)INFO3_SOLID;
    // tiles whose halo lies inside the grid need no wrap / mirror / wall
    // resolution; with FP16 storage their box is one TMA copy (see the FP32 kernel)
    const bool inner = x0 >= 2 && y0 >= 2 && z0 >= 2 && x0 + TX + 2 <= a.nx && y0 + TY + 2 <= a.ny &&
                       z0 + TZ + 2 <= a.nz;
    const bool tma = is_half<S>() && use_tma && inner && (smem_addr(s_rr) & 127u) == 0u;
    if (tma && tid == 0) bar_init(&s_bar);
    // a tile without fluid nodes has nothing to stage or collide
    if (!__syncthreads_or(!(info & INFO3_SOLID))) return;
    if (tid < 2 * Q) s_rate[tid / Q][tid % Q] = a.s[tid / Q][tid % Q];
    if (tma) {
        if (tid == 0) copy_box(&rho_map, s_rr, HN * 8u, x0 - 2, y0 - 2, z0 - 2, &s_bar);
    } else {
        stage_box(a, x0, y0, z0, inner, tid, [&](int q, typename Pair<R>::type v) { s_rr[q] = v; });
    }
    const int fid = (int)((info >> INFO3_FACE_SHIFT) & 7u);
    const int nid = (int)((info >> INFO3_NBR_SHIFT) & 7u);
    // FP16 storage: both components' pulls are in flight while the densities arrive
    S v0[Q], v1[Q];
    float ref0 = 0.f, ref1 = 0.f;
    if (is_half<S>() && fid == 0 && !(info & INFO3_SOLID)) {
        pull_raw<0>(a, x, y, z, n, info, v0);
        pull_raw<1>(a, x, y, z, n, info, v1);
        ref0 = __half2float(a.rref_in[n]);
        ref1 = __half2float(a.rref_in[a.plane + n]);
    }
    if (tma) {
        wait_box(&s_bar, a.status, tid == 0);
    } else {
        __syncthreads();
    }
    if constexpr (is_half<S>()) {
        for (int q = tid; q < HN; q += NT) s_ref[q] = __floats2half2_rn((float)s_rr[q].x, (float)s_rr[q].y);
        __syncthreads();
    }
    if (info & INFO3_SOLID) return;  // solid, or outside the grid
    const int hc = (threadIdx.x + 2) + HX * ((threadIdx.y + 2) + HY * (threadIdx.z + 2));
    auto site = [&](int dx, int dy, int dz) { return s_rr[hc + dx + HX * (dy + HY * dz)]; };
    R f[Q];
    R j[3] = {0, 0, 0};
    int slot = -1;
    auto decode = [&](const S (&v)[Q], float ref) {
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            f[i] = (R)ld_pop(v[i]);
            if constexpr (is_half<S>()) f[i] += ((R)w36_(i) / (R)36) * ref;
        });
    };
    if (!is_half<S>() && fid == 0) pull<0, S, R>(a, x, y, z, info, f);  // loads overlap the stencil below
    R g1[3], g2[3], ad[3];
    stencil_sums<R>(site, g1, g2);
    adhesion_vector<S>(a, n, info, ad);
    const R r1 = s_rr[hc].x, r2 = s_rr[hc].y;
    R F1[3], F2[3];
    forces<R>(a.G, r1, r2, g1, g2, ad, a.body, F1, F2);
    const R rt = r1 + r2;
    if (fid == 0) {
        if constexpr (is_half<S>()) decode(v0, ref0);
        add_j(f, j);
        if constexpr (STASH)
            static_for<0, Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                s_f0[i][tid] = f[i];
            });
        if constexpr (is_half<S>()) decode(v1, ref1);
        else pull<1, S, R>(a, x, y, z, info, f);
        add_j(f, j);
    } else {
        const FaceDev3& Fc = a.face[fid - 1];
        slot = face_slot(Fc, x, y, z);
        R* Fp = a.FpF + (size_t)slot * 6;  // this step's force: next step's inlet, this step's outlet
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            Fp[q] = F1[q];
            Fp[3 + q] = F2[q];
        }
        if (Fc.kind == FACE3_OUTLET) return;  // finished by d3q_outlet_kernel
        const R* ff = a.fface + (size_t)slot * 2 * Q;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            static_for<0, Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                f[i] = ff[k * Q + i];
            });
            add_j(f, j);
        }
    }
    R u[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) u[q] = (j[q] + (R)0.5 * (F1[q] + F2[q])) / rt;
    if (nid != 0) {
        const FaceDev3& Fc = a.face[nid - 1];
        const int ns = face_slot(Fc, x + Fc.o[0], y + Fc.o[1], z + Fc.o[2]);
        R* Fp = a.FpN + (size_t)ns * 6;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            Fp[q] = F1[q];
            Fp[3 + q] = F2[q];
        }
        if (Fc.kind == FACE3_OUTLET) {
            const double sg = (double)(Fc.o[0] + Fc.o[1] + Fc.o[2]);
            R* un = a.unbr + (size_t)ns * 3;
            un[0] = u[0];
            un[1] = u[1];
            un[2] = u[2];
            a.flux[(size_t)ns * 2 + 0] = (double)rt * sg * (double)u[Fc.axis];
            a.flux[(size_t)ns * 2 + 1] = sg * (double)u[Fc.axis];
        }
    }
    if (fid != 0) {  // inlet node: flux term of Q_in
        const FaceDev3& Fc = a.face[fid - 1];
        const double sg = (double)(Fc.o[0] + Fc.o[1] + Fc.o[2]);
        a.flux[(size_t)slot * 2 + 0] = (double)rt * (-sg) * (double)u[Fc.axis];
        a.flux[(size_t)slot * 2 + 1] = 0.0;
    }
    check_store_u<S>(a, n, rt, u);
    // reader densities for FP16 storage: the staged tile (periodic wraps
    // resolved) or this node when the direction is blocked
    auto dest_rho = [&](auto I, int k) -> R {
        constexpr int i = decltype(I)::value;
        const int h = (info & (1u << opp_(i))) ? hc : hc + ex_(i) + HX * (ey_(i) + HY * ez_(i));
        const __half2 r = s_ref[h];
        return k ? __high2float(r) : __low2float(r);
    };
    // no blocked direction (most nodes): constant offsets, no selects
    const bool open = (info & 0x7FFFFu) == 0u;
    auto dest_rho_open = [&](auto I, int k) -> R {
        constexpr int i = decltype(I)::value;
        const __half2 r = s_ref[hc + ex_(i) + HX * (ey_(i) + HY * ez_(i))];
        return k ? __high2float(r) : __low2float(r);
    };
    if constexpr (is_half<S>()) {
        a.rref_out[n] = __float2half_rn(r1);
        a.rref_out[a.plane + n] = __float2half_rn(r2);
    }
    // collide component 1 (still in registers), then component 0 (from the
    // shared-memory copy with FP16 storage, pulled again in FP64): one loop body,
    // so the unrolled collision is in the instruction stream once
#pragma unroll 1
    for (int k = 1; k >= 0; --k) {
        if (k == 0) {
            if (fid == 0) {
                if constexpr (STASH)
                    static_for<0, Q>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        f[i] = s_f0[i][tid];
                    });
                else pull<0, S, R>(a, x, y, z, info, f);
            } else {
                const R* ff = a.fface + (size_t)slot * 2 * Q;
                static_for<0, Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    f[i] = ff[i];
                });
            }
        }
        const R rk = k ? r2 : r1;
        const R fx = k ? F2[0] : F1[0], fy = k ? F2[1] : F1[1], fz = k ? F2[2] : F1[2];
        collide<R>(f, rk, u[0], u[1], u[2], fx, fy, fz, s_rate[k]);
        if (is_half<S>() && open) store_pop<S>(a, k, n, f, dest_rho_open);
        else store_pop<S>(a, k, n, f, dest_rho);
    }
}

// ---- FP32 collision: both components of a node in packed FP32x2 operations ----
__device__ __forceinline__ float2 vc(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, vc(-1.f), a); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ float2 ld_shared2(unsigned addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async4(unsigned dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// The 18 moments of both components that the collision needs besides the
// density, from the populations get(i), with the rows of T written out over the
// sums and differences of opposite pairs: axis pairs (1,2), (3,4), (5,6), edge
// pairs (7,10), (8,9) in xy, (11,14), (12,13) in xz, (15,18), (16,17) in yz.
struct Moments2 {
    float2 e, eps, j[3], q[3], xx, pixx, ww, piww, xy, yz, xz, m[3];
};
template <typename Get>
__device__ __forceinline__ void moments2(Get get, Moments2& M) {
    const float2 f0 = get(0), f1 = get(1), f2 = get(2), f3 = get(3), f4 = get(4), f5 = get(5), f6 = get(6);
    const float2 px = vadd(f1, f2), py = vadd(f3, f4), pz = vadd(f5, f6);
    const float2 dx = vsub(f1, f2), dy = vsub(f3, f4), dz = vsub(f5, f6);
    const float2 f7 = get(7), f10 = get(10), f8 = get(8), f9 = get(9);
    const float2 p7 = vadd(f7, f10), p8 = vadd(f8, f9), d7 = vsub(f7, f10), d8 = vsub(f8, f9);
    const float2 f11 = get(11), f14 = get(14), f12 = get(12), f13 = get(13);
    const float2 p11 = vadd(f11, f14), p12 = vadd(f12, f13), d11 = vsub(f11, f14), d12 = vsub(f12, f13);
    const float2 f15 = get(15), f18 = get(18), f16 = get(16), f17 = get(17);
    const float2 p15 = vadd(f15, f18), p16 = vadd(f16, f17), d15 = vsub(f15, f18), d16 = vsub(f16, f17);
    const float2 sxy = vadd(p7, p8), sxz = vadd(p11, p12), syz = vadd(p15, p16);
    const float2 sa = vadd(px, vadd(py, pz)), se = vadd(vadd(sxy, sxz), syz);
    M.e = vfma(vc(-30.f), f0, vfma(vc(-11.f), sa, vmul(vc(8.f), se)));
    M.eps = vfma(vc(12.f), f0, vfma(vc(-4.f), sa, se));
    const float2 exy = vsub(d7, d8), exz = vsub(d11, d12), eyx = vadd(d7, d8), eyz = vsub(d15, d16),
                 ezx = vadd(d11, d12), ezy = vadd(d15, d16);
    const float2 jx = vadd(exy, exz), jy = vadd(eyx, eyz), jz = vadd(ezx, ezy);
    M.j[0] = vadd(dx, jx);
    M.j[1] = vadd(dy, jy);
    M.j[2] = vadd(dz, jz);
    M.q[0] = vfma(vc(-4.f), dx, jx);
    M.q[1] = vfma(vc(-4.f), dy, jy);
    M.q[2] = vfma(vc(-4.f), dz, jz);
    const float2 ax = vsub(vmul(vc(2.f), px), vadd(py, pz)), exx = vfma(vc(-2.f), syz, vadd(sxy, sxz));
    M.xx = vadd(ax, exx);
    M.pixx = vfma(vc(-2.f), ax, exx);
    const float2 aw = vsub(py, pz), ew = vsub(sxy, sxz);
    M.ww = vadd(aw, ew);
    M.piww = vfma(vc(-2.f), aw, ew);
    M.xy = vsub(p7, p8);
    M.yz = vsub(p15, p16);
    M.xz = vsub(p11, p12);
    M.m[0] = vsub(exy, exz);
    M.m[1] = vsub(eyz, eyx);
    M.m[2] = vsub(ezx, ezy);
}

// Eq. 1 as in collide(), from the moments; put(i, value to add) per direction.
// s: rates of (e, eps, j, q, nu), the values the 19 diagonal entries take (pi
// shares eps, m shares q).
template <typename Put>
__device__ __forceinline__ void collide2(const Moments2& M, float2 r, float ux, float uy, float uz,
                                         const float2 (&F)[3], const float2 (&s)[5], Put put) {
    const float2 U = vc(ux), V = vc(uy), W = vc(uz);
    const float2 Fx = F[0], Fy = F[1], Fz = F[2];
    const float xx = ux * ux, yy = uy * uy, zz = uz * uz, uu = xx + yy + zz;
    const float2 uF = vfma(U, Fx, vfma(V, Fy, vmul(W, Fz)));
    const float2 half = vc(0.5f);
    float2 h[5], ns[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        h[q] = vfma(vc(-0.5f), s[q], vc(1.f));
        ns[q] = vmul(vc(-1.f), s[q]);
    }
    // g_r = (-s (m - m^eq) + (1 - s/2) F_m) / |row|^2
    const float2 ge = vmul(vc(1.f / 2394.f), vfma(ns[0], vsub(M.e, vmul(r, vc(19.f * uu - 11.f))),
                                                  vmul(h[0], vmul(vc(38.f), uF))));
    const float2 gp = vmul(vc(1.f / 252.f), vfma(ns[1], vsub(M.eps, vmul(r, vc(3.f - 5.5f * uu))),
                                                 vmul(h[1], vmul(vc(-11.f), uF))));
    const float2 rux = vmul(r, U), ruy = vmul(r, V), ruz = vmul(r, W);
    const float2 c10 = vc(0.1f), c40 = vc(1.f / 40.f), t23 = vc(2.f / 3.f);
    const float2 gjx = vmul(c10, vfma(ns[2], vsub(M.j[0], rux), vmul(h[2], Fx)));
    const float2 gjy = vmul(c10, vfma(ns[2], vsub(M.j[1], ruy), vmul(h[2], Fy)));
    const float2 gjz = vmul(c10, vfma(ns[2], vsub(M.j[2], ruz), vmul(h[2], Fz)));
    // q^eq = -2/3 rho u, its forcing -2/3 F
    const float2 hq = vmul(vmul(vc(-1.f), t23), h[3]);
    const float2 gqx = vmul(c40, vfma(ns[3], vfma(t23, rux, M.q[0]), vmul(hq, Fx)));
    const float2 gqy = vmul(c40, vfma(ns[3], vfma(t23, ruy, M.q[1]), vmul(hq, Fy)));
    const float2 gqz = vmul(c40, vfma(ns[3], vfma(t23, ruz, M.q[2]), vmul(hq, Fz)));
    // 3p_xx and 3pi_xx (equilibrium and forcing of pi: -1/2 of p's)
    const float2 qxx = vmul(r, vc(2.f * xx - yy - zz));
    const float2 fxx = vmul(vc(2.f), vsub(vmul(vmul(vc(2.f), U), Fx), vfma(V, Fy, vmul(W, Fz))));
    const float2 gxx = vmul(vc(1.f / 36.f), vfma(ns[4], vsub(M.xx, qxx), vmul(h[4], fxx)));
    const float2 gyx = vmul(vc(1.f / 72.f), vfma(ns[1], vfma(half, qxx, M.pixx), vmul(h[1], vmul(vc(-0.5f), fxx))));
    // p_ww and pi_ww
    const float2 qww = vmul(r, vc(yy - zz)), fww = vmul(vc(2.f), vsub(vmul(V, Fy), vmul(W, Fz)));
    const float2 gww = vmul(vc(1.f / 12.f), vfma(ns[4], vsub(M.ww, qww), vmul(h[4], fww)));
    const float2 gyw = vmul(vc(1.f / 24.f), vfma(ns[1], vfma(half, qww, M.piww), vmul(h[1], vmul(vc(-0.5f), fww))));
    // p_xy, p_yz, p_xz
    const float2 c4 = vc(0.25f);
    const float2 gxy = vmul(c4, vfma(ns[4], vsub(M.xy, vmul(rux, V)), vmul(h[4], vfma(U, Fy, vmul(V, Fx)))));
    const float2 gyz = vmul(c4, vfma(ns[4], vsub(M.yz, vmul(ruy, W)), vmul(h[4], vfma(V, Fz, vmul(W, Fy)))));
    const float2 gxz = vmul(c4, vfma(ns[4], vsub(M.xz, vmul(rux, W)), vmul(h[4], vfma(U, Fz, vmul(W, Fx)))));
    // m_x, m_y, m_z (no equilibrium, no forcing)
    const float2 n8 = vmul(vc(0.125f), ns[3]);
    const float2 gmx = vmul(n8, M.m[0]), gmy = vmul(n8, M.m[1]), gmz = vmul(n8, M.m[2]);
    // back: f_i += even + odd, f_ibar += even - odd
    auto both = [&](int i, int o, float2 ev, float2 od) {
        put(i, vadd(ev, od));
        put(o, vsub(ev, od));
    };
    put(0, vfma(vc(-30.f), ge, vmul(vc(12.f), gp)));
    const float2 ea = vfma(vc(-11.f), ge, vmul(vc(-4.f), gp)), ee = vfma(vc(8.f), ge, gp);
    const float2 axx = vfma(vc(-2.f), gyx, gxx), aww = vfma(vc(-2.f), gyw, gww);
    both(1, 2, vfma(vc(2.f), axx, ea), vfma(vc(-4.f), gqx, gjx));
    const float2 eb = vsub(ea, axx);
    both(3, 4, vadd(eb, aww), vfma(vc(-4.f), gqy, gjy));
    both(5, 6, vsub(eb, aww), vfma(vc(-4.f), gqz, gjz));
    const float2 Jx = vadd(gjx, gqx), Jy = vadd(gjy, gqy), Jz = vadd(gjz, gqz);
    const float2 bxx = vadd(gxx, gyx), bww = vadd(gww, gyw), e1 = vadd(ee, bxx);
    {
        const float2 A = vadd(Jx, gmx), B = vsub(Jy, gmy), e = vadd(e1, bww);
        both(7, 10, vadd(e, gxy), vadd(A, B));
        both(8, 9, vsub(e, gxy), vsub(B, A));
    }
    {
        const float2 A = vsub(Jx, gmx), B = vadd(Jz, gmz), e = vsub(e1, bww);
        both(11, 14, vadd(e, gxz), vadd(A, B));
        both(12, 13, vsub(e, gxz), vsub(B, A));
    }
    {
        const float2 A = vadd(Jy, gmy), B = vsub(Jz, gmz), e = vfma(vc(-2.f), bxx, ee);
        both(15, 18, vadd(e, gyz), vadd(A, B));
        both(16, 17, vsub(e, gyz), vsub(B, A));
    }
}

// FP32: the same step as d3q_collide_kernel with both components of a node in
// the two lanes of packed FP32x2 instructions (half the instructions).  All 38
// pulls of a node go straight to shared memory (cp.async) before the density
// box is waited for, and are read from there twice, for the moments and for the
// result: 80 registers and three CTAs of 256 per SM instead of two at 126 with
// the populations in registers (265 against 277 us on the 512x96x96 co-flow
// device; one component after the other, 64 registers: 330).  The rest is load
// latency and shared-memory throughput (l1tex 58 %, DRAM 51 %).
__global__ void __launch_bounds__(Tile3<float>::NT, Tile3<float>::MIN_BLOCKS)
    d3q_collide_f32_kernel(const __grid_constant__ D3Args<float> a, const __grid_constant__ CUtensorMap rho_map,
                           int use_tma, int zblock) {
    constexpr int TZ = Tile3<float>::TZ, HN = Tile3<float>::HN, NT = Tile3<float>::NT;
    // (rho_1, rho_2) of the tile and its halo, psi = 0 at solids; 128-byte
    // aligned: an interior tile receives it as one tensor copy.  Behind it the
    // pulled populations [Q][NT] as component pairs.
    extern __shared__ __align__(128) unsigned char s_dyn[];
    float2* s_rr = reinterpret_cast<float2*>(s_dyn);
    __shared__ __align__(8) unsigned long long s_bar;
    // from the last z on: the pull kernel has just read those planes (L2), and the
    // next one starts on the planes this kernel writes last (co-flow 250x64x64
    // 112.7 us per step in ascending order, 108.4 in this one; 512x96x96 400, 397)
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = (zblock + (int)(gridDim.z - 1 - blockIdx.z)) * TZ;
    const int tid = threadIdx.x + TX * (threadIdx.y + TY * threadIdx.z);
    const unsigned s_f = smem_addr(s_rr + HN) + 8u * (unsigned)tid;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    const bool in_grid = x < a.nx && y < a.ny && z < a.nz;
    const long long n = in_grid ? node_index(a, x, y, z) : 0;
    const uint32_t info = in_grid ? a.info[n] : (uint32_t)INFO3_SOLID;
    // tiles whose halo lies inside the grid need no wrap / mirror / wall
    // resolution; their box comes as one TMA copy (x0 - 2 is even: an 8-byte
    // element start on a 16-byte boundary).  The block-uniform test keeps a
    // misaligned destination on the load path.
    const bool inner = x0 >= 2 && y0 >= 2 && z0 >= 2 && x0 + TX + 2 <= a.nx && y0 + TY + 2 <= a.ny &&
                       z0 + TZ + 2 <= a.nz;
    const bool tma = use_tma && inner && (smem_addr(s_rr) & 127u) == 0u;
    if (tma && tid == 0) bar_init(&s_bar);
    // a tile without fluid nodes has nothing to stage or collide
    if (!__syncthreads_or(!(info & INFO3_SOLID))) return;
    if (tma) {
        if (tid == 0) copy_box(&rho_map, s_rr, HN * 8u, x0 - 2, y0 - 2, z0 - 2, &s_bar);
    } else {
        stage_box(a, x0, y0, z0, inner, tid, [&](int q, float2 v) { s_rr[q] = v; });
    }
    const int fid = (int)((info >> INFO3_FACE_SHIFT) & 7u);
    const int nid = (int)((info >> INFO3_NBR_SHIFT) & 7u);
    // all 38 pulls go to shared memory while the densities arrive
    int slot = -1;
    if (!(info & INFO3_SOLID)) {
        if (fid == 0) {
            pull_sources<0, 2>(a, x, y, z, n, info,
                                [&](int k, int i, const float* p) { cp_async4(s_f + 8u * NT * i + 4u * k, p); });
        } else {
            slot = face_slot(a.face[fid - 1], x, y, z);
            const float* ff = a.fface + (size_t)slot * 2 * Q;
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int i = 0; i < Q; ++i) cp_async4(s_f + 8u * NT * i + 4u * k, ff + k * Q + i);
        }
    }
    if (tma) {
        wait_box(&s_bar, a.status, tid == 0);
    } else {
        __syncthreads();
    }
    if (info & INFO3_SOLID) return;  // solid, or outside the grid
    const int hc = (threadIdx.x + 2) + HX * ((threadIdx.y + 2) + HY * (threadIdx.z + 2));
    const float2 r = s_rr[hc];
    float g1[3], g2[3], ad[3];
    stencil_sums<float>([&](int dx, int dy, int dz) { return s_rr[hc + dx + HX * (dy + HY * dz)]; }, g1, g2);
    adhesion_vector<float>(a, n, info, ad);
    const float rt = r.x + r.y, inv = 1.f / rt;
    float2 F[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float2 t = vfma(make_float2(-a.G[1], -a.G[2]), vc(ad[q]), vmul(vc(-a.G[0]), make_float2(g2[q], g1[q])));
        F[q] = vmul(r, vadd(t, vc(a.body[q] * inv)));
    }
    if (fid != 0) {
        const FaceDev3& Fc = a.face[fid - 1];
        float* Fp = a.FpF + (size_t)slot * 6;  // this step's force: next step's inlet, this step's outlet
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            Fp[q] = F[q].x;
            Fp[3 + q] = F[q].y;
        }
        if (Fc.kind == FACE3_OUTLET) {  // finished by d3q_outlet_kernel
            asm volatile("cp.async.wait_all;" ::: "memory");  // no copy outlives its thread
            return;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    auto pop = [&](int i) { return ld_shared2(s_f + 8u * NT * i); };
    Moments2 M;
    moments2(pop, M);
    float u[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float2 t = vfma(vc(0.5f), F[q], M.j[q]);
        u[q] = (t.x + t.y) * inv;
    }
    if (nid != 0) {
        const FaceDev3& Fc = a.face[nid - 1];
        const int ns = face_slot(Fc, x + Fc.o[0], y + Fc.o[1], z + Fc.o[2]);
        float* Fp = a.FpN + (size_t)ns * 6;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            Fp[q] = F[q].x;
            Fp[3 + q] = F[q].y;
        }
        if (Fc.kind == FACE3_OUTLET) {
            const double sg = (double)(Fc.o[0] + Fc.o[1] + Fc.o[2]);
            const float ua = Fc.axis == 0 ? u[0] : (Fc.axis == 1 ? u[1] : u[2]);
            float* un = a.unbr + (size_t)ns * 3;
            un[0] = u[0];
            un[1] = u[1];
            un[2] = u[2];
            a.flux[(size_t)ns * 2 + 0] = (double)rt * sg * (double)ua;
            a.flux[(size_t)ns * 2 + 1] = sg * (double)ua;
        }
    }
    if (fid != 0) {  // inlet node: flux term of Q_in
        const FaceDev3& Fc = a.face[fid - 1];
        const double sg = (double)(Fc.o[0] + Fc.o[1] + Fc.o[2]);
        const float ua = Fc.axis == 0 ? u[0] : (Fc.axis == 1 ? u[1] : u[2]);
        a.flux[(size_t)slot * 2 + 0] = (double)rt * (-sg) * (double)ua;
        a.flux[(size_t)slot * 2 + 1] = 0.0;
    }
    check_store_u<float>(a, n, rt, u);
    const float2 s[5] = {make_float2(a.s[0][1], a.s[1][1]), make_float2(a.s[0][2], a.s[1][2]),
                         make_float2(a.s[0][3], a.s[1][3]), make_float2(a.s[0][4], a.s[1][4]),
                         make_float2(a.s[0][9], a.s[1][9])};
    const unsigned off = (unsigned)n * 4u;
    collide2(M, r, u[0], u[1], u[2], F, s, [&](int i, float2 d) {
        const float2 v = vadd(pop(i), d);
        st_at(a.dst[0][i], off, v.x);
        st_at(a.dst[1][i], off, v.y);
    });
}

// One thread per outlet slot: the outlet node's velocity with the normal
// component chi times that of its inward neighbour (Eq. 22), the collision.
template <typename S>
__global__ void __launch_bounds__(128) d3q_outlet_kernel(D3Args<S> a) {
    using R = typename Store<S>::R;
    int fid, c[3];
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (!slot_node(a, slot, fid, c)) return;
    const FaceDev3& Fc = a.face[fid];
    if (Fc.kind != FACE3_OUTLET) return;
    const long long n = node_index(a, c[0], c[1], c[2]);
    const R r1 = a.rho[2 * n], r2 = a.rho[2 * n + 1], rt = r1 + r2;
    const R* Fp = a.FpF + (size_t)slot * 6;
    const R F1[3] = {Fp[0], Fp[1], Fp[2]}, F2[3] = {Fp[3], Fp[4], Fp[5]};
    const R* ff = a.fface + (size_t)slot * 2 * Q;
    R f[Q], j[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            f[i] = ff[k * Q + i];
        });
        add_j(f, j);
    }
    R u[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) u[q] = (j[q] + (R)0.5 * (F1[q] + F2[q])) / rt;
    if (Fc.chi) u[Fc.axis] = (R)a.scal_in[SC3_CHI] * a.unbr[(size_t)slot * 3 + Fc.axis];
    check_store_u<S>(a, n, rt, u);
    const uint32_t info = a.info[n];
    auto dest_rho = [&](auto I, int k) -> R {
        constexpr int i = decltype(I)::value;
        long long m = n;
        if (!(info & (1u << opp_(i)))) m = site_index(a, c[0] + ex_(i), c[1] + ey_(i), c[2] + ez_(i));
        return half_round(a.rho[2 * m + k]);
    };
    if constexpr (is_half<S>()) {
        a.rref_out[n] = __float2half_rn(r1);
        a.rref_out[a.plane + n] = __float2half_rn(r2);
    }
    collide<R>(f, r2, u[0], u[1], u[2], F2[0], F2[1], F2[2], a.s[1]);
    store_pop<S>(a, 1, n, f, dest_rho);
    static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        f[i] = ff[i];
    });
    collide<R>(f, r1, u[0], u[1], u[2], F1[0], F1[1], F1[2], a.s[0]);
    store_pop<S>(a, 0, n, f, dest_rho);
}

// ---- kernel C: lambda and chi from the face flux terms (fixed order) -------
// One block of 1024 threads; each thread owns a fixed set of slots and the
// tree below has a fixed shape, so the sums are deterministic.  Slots of
// solid face positions hold the zeros they were created with.
constexpr int RED = 1024;
template <typename S>
__global__ void __launch_bounds__(RED) d3q_reduce_kernel(D3Args<S> a) {
    __shared__ double s_in[RED], s_out[RED], s_u[RED];
    double qin = 0.0, qout = 0.0, us = 0.0;
    const double2* fl = reinterpret_cast<const double2*>(a.flux);
    for (int f = 0; f < a.nfaces; ++f) {
        const FaceDev3& F = a.face[f];
        const bool inlet = F.kind == FACE3_INLET;
#pragma unroll 4
        for (int q = threadIdx.x; q < F.count; q += RED) {
            const double2 v = fl[F.base + q];
            if (inlet) qin += v.x;
            else {
                qout += v.x;
                us += v.y;
            }
        }
    }
    s_in[threadIdx.x] = qin;
    s_out[threadIdx.x] = qout;
    s_u[threadIdx.x] = us;
    __syncthreads();
    for (int w = RED / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            s_in[threadIdx.x] += s_in[threadIdx.x + w];
            s_out[threadIdx.x] += s_out[threadIdx.x + w];
            s_u[threadIdx.x] += s_u[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double* sc = a.scal_out;
        const double Qi = s_in[0], Qo = s_out[0];
        sc[SC3_QIN] = Qi;
        sc[SC3_QOUT] = Qo;
        if (a.out_count > 0) {
            const double lam = s_u[0] / (double)a.out_count;
            sc[SC3_UMEAN] = lam;
            sc[SC3_LAMBDA] = lam > 0.0 ? lam : 0.0;
            sc[SC3_CHI] = (!a.have_inlet || fabs(Qo) < 1e-14) ? 1.0 : Qi / Qo;
        } else {
            sc[SC3_UMEAN] = a.scal_in[SC3_UMEAN];
            sc[SC3_LAMBDA] = a.scal_in[SC3_LAMBDA];
            sc[SC3_CHI] = a.scal_in[SC3_CHI];
        }
    }
}

// ---- diagnostics: FP64 masses over fluid nodes and the largest |u|^2 ------
template <typename S>
__global__ void __launch_bounds__(256) d3q_mass_kernel(const S* __restrict__ f, const uint32_t* __restrict__ info,
                                                       const typename Store<S>::R* __restrict__ umac,
                                                       const __half* __restrict__ rref, int nx, int ny, int nz,
                                                       int pitch, long long plane, double* __restrict__ partial) {
    __shared__ double s0[256], s1[256], s2[256];
    double m0 = 0.0, m1 = 0.0, u2 = 0.0;
    const long long total = (long long)nx * ny * nz;
    for (long long q = (long long)blockIdx.x * 256 + threadIdx.x; q < total; q += (long long)gridDim.x * 256) {
        const int x = (int)(q % nx);
        const long long yz = q / nx;
        const int y = (int)(yz % ny), z = (int)(yz / ny);
        const long long n = yz * pitch + x;
        const uint32_t inf = info[n];
        if (inf & INFO3_SOLID) continue;
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            double v0 = (double)ld_pop(f[(size_t)i * plane + n]);
            double v1 = (double)ld_pop(f[(size_t)(Q + i) * plane + n]);
            if constexpr (is_half<S>()) {
                // decode with the reference of the node that will pull the value
                long long m = n;
                if (!(inf & (1u << opp_(i)))) {
                    const int xs = ex_(i) ? wrap(x + ex_(i), nx) : x;
                    const int ys = ey_(i) ? wrap(y + ey_(i), ny) : y;
                    const int zs = ez_(i) ? wrap(z + ez_(i), nz) : z;
                    m = ((long long)zs * ny + ys) * pitch + xs;
                }
                const double w = (double)w36_(i) / 36.0;
                v0 += w * (double)__half2float(rref[m]);
                v1 += w * (double)__half2float(rref[plane + m]);
            }
            m0 += v0;
            m1 += v1;
        });
        const double ux = (double)umac[n], uy = (double)umac[plane + n], uz = (double)umac[2 * plane + n];
        u2 = fmax(u2, ux * ux + uy * uy + uz * uz);
    }
    s0[threadIdx.x] = m0;
    s1[threadIdx.x] = m1;
    s2[threadIdx.x] = u2;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            s0[threadIdx.x] += s0[threadIdx.x + w];
            s1[threadIdx.x] += s1[threadIdx.x + w];
            s2[threadIdx.x] = fmax(s2[threadIdx.x], s2[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[blockIdx.x * 3] = s0[0];
        partial[blockIdx.x * 3 + 1] = s1[0];
        partial[blockIdx.x * 3 + 2] = s2[0];
    }
}

// Macroscopic fields for a reader on the device (one pass, 20 bytes in and out
// per node).  Reordering them on the host between two copies made 50 steps of
// 512x96x96 with one read take 45.7 ms; with this kernel they take 25.3 ms.
template <typename R>
__global__ void __launch_bounds__(256) d3q_macros_kernel(const R* __restrict__ rho_pairs, const R* __restrict__ umac,
                                                         const uint32_t* __restrict__ info, int nx, long long rows,
                                                         int pitch, long long plane,
                                                         const unsigned* __restrict__ status,
                                                         float* __restrict__ rho, float* __restrict__ u,
                                                         unsigned* __restrict__ status_out) {
    const unsigned st = *status;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) *status_out = st;
    if (st) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nx) return;
    const long long N = rows * nx;
    for (long long row = (long long)blockIdx.y * blockDim.y + threadIdx.y; row < rows;
         row += (long long)gridDim.y * blockDim.y) {
        const long long n = row * pitch + x, h = row * nx + x;
        const bool solid = (info[n] & INFO3_SOLID) != 0;
        const typename Pair<R>::type r = reinterpret_cast<const typename Pair<R>::type*>(rho_pairs)[n];
        rho[h] = solid ? 0.f : (float)r.x;
        rho[N + h] = solid ? 0.f : (float)r.y;
#pragma unroll
        for (int q = 0; q < 3; ++q) u[q * N + h] = solid ? 0.f : (float)umac[q * plane + n];
    }
}

template <typename R>
cudaError_t launch_macros(const R* rho_pairs, const R* umac, const uint32_t* info, int nx, int ny, int nz, int pitch,
                          long long plane, const unsigned* status, float* rho, float* u, unsigned* status_out,
                          cudaStream_t st) {
    const long long rows = (long long)ny * nz;
    const dim3 blk(64, 4);
    const dim3 grid((unsigned)((nx + 63) / 64), (unsigned)((rows + 3) / 4 < 65535 ? (rows + 3) / 4 : 65535));
    d3q_macros_kernel<R><<<grid, blk, 0, st>>>(rho_pairs, umac, info, nx, rows, pitch, plane, status, rho, u,
                                               status_out);
    return cudaGetLastError();
}

constexpr int GRID_Z = 65535;  // largest z extent of a launch grid: longer grids take several launches

template <typename S>
static cudaError_t launch_pull(const D3Args<S>& a, cudaStream_t st) {
    const dim3 blk(32, 4, 2);
    for (int z = 0; z < a.nz; z += GRID_Z) {
        const dim3 grd((a.nx + 31) / 32, (a.ny + 3) / 4, std::min(GRID_Z, a.nz - z));
        d3q_pull_kernel<S><<<grd, blk, 0, st>>>(a, z);
    }
    return cudaGetLastError();
}

constexpr size_t COLLIDE_F32_SMEM = (size_t)(Tile3<float>::HN + Q * Tile3<float>::NT) * sizeof(float2);

cudaError_t prepare_kernels() {
    return cudaFuncSetAttribute(d3q_collide_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)COLLIDE_F32_SMEM);
}

template <typename S>
static cudaError_t launch_collide(const D3Args<S>& a, const CUtensorMap* rho_map, cudaStream_t st) {
    static const CUtensorMap kNoMap{};
    constexpr int TZ = Tile3<S>::TZ;
    const dim3 blk(TX, TY, TZ);
    const int nzb = (a.nz + TZ - 1) / TZ;
    for (int z = 0; z < nzb; z += GRID_Z) {
        const dim3 grd((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY, std::min(GRID_Z, nzb - z));
        if constexpr (std::is_same<S, float>::value)
            d3q_collide_f32_kernel<<<grd, blk, COLLIDE_F32_SMEM, st>>>(a, rho_map ? *rho_map : kNoMap, rho_map ? 1 : 0, z);
        else
            d3q_collide_kernel<S><<<grd, blk, 0, st>>>(a, rho_map ? *rho_map : kNoMap, rho_map ? 1 : 0, z);
    }
    return cudaGetLastError();
}

constexpr int FACE_NT = 64;  // threads of a face block: few long threads, spread over many SMs
static int face_blocks(int slots) { return (slots + FACE_NT - 1) / FACE_NT; }

template <typename S>
cudaError_t launch_step(const D3Args<S>& a, const CUtensorMap* rho_map, cudaStream_t st, cudaEvent_t mid_a,
                        cudaEvent_t mid_b) {
    cudaError_t e = launch_pull(a, st);
    if (e != cudaSuccess) return e;
    if (a.nface_slots > 0) {
        d3q_face_pull_kernel<S><<<face_blocks(a.nface_slots), FACE_NT, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (mid_a) cudaEventRecord(mid_a, st);
    if ((e = launch_collide(a, rho_map, st)) != cudaSuccess) return e;
    if (mid_b) cudaEventRecord(mid_b, st);
    if (a.nface_slots > 0) {
        d3q_outlet_kernel<S><<<face_blocks(a.nface_slots), FACE_NT, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        d3q_reduce_kernel<S><<<1, RED, 0, st>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

// Branch order.  The face pulls of a step need the previous step's collision,
// outlet and reduction; the interior pulls the collision and outlet only; the
// collision both pulls.  The reduction reads the flux terms, which the next
// collision (after the next face pulls, hence after it) overwrites.
template <typename S>
cudaError_t launch_step_forked(const D3Args<S>& a, const CUtensorMap* rho_map, cudaStream_t st, cudaStream_t side,
                               const cudaEvent_t (&ev)[3]) {
    cudaError_t e = cudaSuccess;
    const bool faces = a.nface_slots > 0;
    if (faces) {
        d3q_face_pull_kernel<S><<<face_blocks(a.nface_slots), FACE_NT, 0, side>>>(a);
        if ((e = cudaGetLastError()) == cudaSuccess) e = cudaEventRecord(ev[1], side);
    }
    if (e == cudaSuccess) e = launch_pull(a, st);
    if (faces && e == cudaSuccess) e = cudaStreamWaitEvent(st, ev[1], 0);
    if (e == cudaSuccess) e = launch_collide(a, rho_map, st);
    if (!faces || e != cudaSuccess) return e;
    if ((e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
    d3q_outlet_kernel<S><<<face_blocks(a.nface_slots), FACE_NT, 0, st>>>(a);
    if ((e = cudaGetLastError()) == cudaSuccess) e = cudaEventRecord(ev[0], st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ev[2], 0);
    if (e != cudaSuccess) return e;
    d3q_reduce_kernel<S><<<1, RED, 0, side>>>(a);
    if ((e = cudaGetLastError()) == cudaSuccess) e = cudaStreamWaitEvent(side, ev[0], 0);
    return e;
}

template <typename S>
cudaError_t launch_mass(const S* f, const uint32_t* info, const typename Real<S>::type* umac, const __half* rref,
                        int nx, int ny, int nz, int pitch, long long plane, double* partial, int nblocks,
                        cudaStream_t st) {
    d3q_mass_kernel<S><<<nblocks, 256, 0, st>>>(f, info, umac, rref, nx, ny, nz, pitch, plane, partial);
    return cudaGetLastError();
}

template cudaError_t launch_step<float>(const D3Args<float>&, const CUtensorMap*, cudaStream_t, cudaEvent_t,
                                          cudaEvent_t);
template cudaError_t launch_step<double>(const D3Args<double>&, const CUtensorMap*, cudaStream_t, cudaEvent_t,
                                          cudaEvent_t);
template cudaError_t launch_step<__half>(const D3Args<__half>&, const CUtensorMap*, cudaStream_t, cudaEvent_t,
                                          cudaEvent_t);
template cudaError_t launch_step_forked<float>(const D3Args<float>&, const CUtensorMap*, cudaStream_t, cudaStream_t,
                                               const cudaEvent_t (&)[3]);
template cudaError_t launch_step_forked<double>(const D3Args<double>&, const CUtensorMap*, cudaStream_t,
                                                cudaStream_t, const cudaEvent_t (&)[3]);
template cudaError_t launch_step_forked<__half>(const D3Args<__half>&, const CUtensorMap*, cudaStream_t,
                                                cudaStream_t, const cudaEvent_t (&)[3]);
template cudaError_t launch_macros<float>(const float*, const float*, const uint32_t*, int, int, int, int, long long,
                                           const unsigned*, float*, float*, unsigned*, cudaStream_t);
template cudaError_t launch_macros<double>(const double*, const double*, const uint32_t*, int, int, int, int,
                                            long long, const unsigned*, float*, float*, unsigned*, cudaStream_t);
template cudaError_t launch_mass<float>(const float*, const uint32_t*, const float*, const __half*, int, int, int,
                                        int, long long, double*, int, cudaStream_t);
template cudaError_t launch_mass<double>(const double*, const uint32_t*, const double*, const __half*, int, int, int,
                                         int, long long, double*, int, cudaStream_t);
template cudaError_t launch_mass<__half>(const __half*, const uint32_t*, const float*, const __half*, int, int, int,
                                         int, long long, double*, int, cudaStream_t);

}  // namespace lbm3
