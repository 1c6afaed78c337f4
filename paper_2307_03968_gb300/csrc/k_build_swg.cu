// GPU construction of the V-EFIE H-Matrix of an inhomogeneous dielectric body
// from a tetrahedral mesh (arxiv 2307.03968 §II eq. 4, SWG basis [21]).
//
// Unknowns: one SWG function per face, D = eps0 sum_n x_n f_n; on T+
// f = +(a/3V)(r - v), on T- f = -(a/3V)(r - v), v the vertex opposite the
// face; boundary faces carry the T+ half only.  Contrast kappa = 1 - 1/eps_r
// per tetrahedron.  Eq. 4 (E_inc = D/eps + jwA + grad phi, polarisation current
// J = jw kappa D) tested with kappa f_m gives the complex-symmetric entries
//   Z_mn = Int (kappa/eps_r) f_m . f_n dV - k^2 Int Int kappa f_m . kappa' f_n' G
//          + Int Int q_m q_n' G,
// q the charge of kappa f: -kappa s a / V inside each tetrahedron (s = +-1 on
// T+/T-) and kappa(T+) - kappa(T-) on the function's own face (kappa(T+) on a
// boundary face).  The symmetric form is what makes the half storage of §III
// apply to the volume equation.
//
// Quadrature: 4-point degree-2 rule on tetrahedra, 7-point degree-5 rule on
// triangles.  Element pairs whose centroids are closer than 2 x the larger
// maximum edge length get the 1/R part of G analytically over the inner
// element: over a triangle from the edge form of the potential integrals
// (Wilton et al. 1984, Graglia 1993), over a tetrahedron by the divergence
// theorem, Int_T 1/R dV' = 1/2 sum_f ((p_f - r) . n_f) Int_f 1/R dS' and
// Int_T (r' - r)/R dV' = sum_f n_f Int_f R dS' with outward face normals n_f.
// Coordinates are taken relative to a vertex of the column face.  The near
// blocks (complex64, k_fill_swg) take the quadrature in FP32 but the analytic singular
// terms in FP64: the four tetrahedron pairs of one function pair cancel like a
// dipole-dipole interaction, which turns the ~1e-6 FP32 error of the edge
// formulas two or three element sizes away into ~1e-4 of the entry.  The leaf
// self blocks are filled entirely in FP64.
#include "k_assemble.cuh"

namespace hm {
namespace {

constexpr int NQT = 4;    // tetrahedron rule: barycentric (a,b,b,b) and permutations, weights 1/4
constexpr int NQF = 7;    // triangle rule (degree 5)
constexpr double EXTRACT_FACTOR = 2.0;
constexpr double INV4PI = 0.25 / 3.14159265358979323846;

__constant__ double c_fw[NQF];

constexpr int FGEO = 31;                 // P[3][3], n[3], dir[3][3], out[3][3], 2 area
constexpr int TGEO = 12 + 4 * (3 + 9 + 1) + 6 * 4;   // P[4][3]; faces: n[3], out[3][3], 2 area; edges: dir[3], length

struct VGeo {
    const double *vtx;      // nv x 3
    const int32_t *tet;     // nt x 4
    const double *tqp;      // nt x NQT x 3
    const double *tcen;     // nt x 3
    const double *thmax;    // nt
    const double *tvol;     // nt
    const double *kappa;    // nt
    const double *epsr;     // nt
    const int32_t *fv;      // nf x 3 (ascending)
    const int32_t *ftet;    // nf x 2 (T+, T- or -1)
    const int32_t *ffree;   // nf x 2
    const double *fqp;      // nf x NQF x 3
    const double *fcen;     // nf x 3
    const double *fhmax;    // nf
    const double *farea;    // nf
    const double *fqs;      // nf surface charge kappa(T+) - kappa(T-)
    const int32_t *perm;    // tree position -> original face index
    double k;
    static constexpr int PARTS = 1;
    static constexpr bool BLOCK_FILL = true;
    // for the near fill by blocks (k_fill_swg)
    const float2 *vtx32, *tqp32, *fqp32;   // the points relative to the mesh's middle, as pairs of floats (hi, lo)
    const double *fgeo;     // nf x FGEO: vertices, unit normal away from T+'s free vertex, per edge direction and outward in-plane normal
    const double *tgeo;     // nt x TGEO: vertices; per face (opposite vertex a): outward normal, per edge of the face its outward in-plane normal; the 6 edge directions and lengths
    hm_status fill_near(const std::vector<FillJob> &jobs, float2 *pool, TmpBuffers &tmp, cudaStream_t s) const;
    template <class R> __device__ CX<R> entry(int m, int n) const;
};

// Singular-extraction predicate in FP64 without contractions (the same decision
// as any IEEE FP64 evaluation of |c_a - c_b|^2 < (2 max(h_a, h_b))^2).
__device__ __forceinline__ bool near_pair(const double *ca, double ha, const double *cb, double hb)
{
    const double dx = __dsub_rn(ca[0], cb[0]);
    const double dy = __dsub_rn(ca[1], cb[1]);
    const double dz = __dsub_rn(ca[2], cb[2]);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double h = ha > hb ? ha : hb;
    const double lim = __dmul_rn(EXTRACT_FACTOR, h);
    return d2 < __dmul_rn(lim, lim);
}

template <class R> __device__ __forceinline__ void loc(const double *p, const double *o, R out[3])
{
    out[0] = (R)(p[0] - o[0]);
    out[1] = (R)(p[1] - o[1]);
    out[2] = (R)(p[2] - o[2]);
}

template <class R> __device__ __forceinline__ R dot(const R a[3], const R b[3])
{
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// G (extract = false) or its smooth part G - 1/(4 pi R) (extract = true)
template <class R> __device__ __forceinline__ CX<R> green(R k, R Rr, bool extract)
{
    const R inv4pi = (R)(0.25 / 3.14159265358979323846);
    if (extract) {
        if (Rr < (R)1e-12) return CX<R>{0, -k * inv4pi};
        const R sh = sinR((R)0.5 * k * Rr);
        return CX<R>{-(R)2 * sh * sh * inv4pi / Rr, -sinR(k * Rr) * inv4pi / Rr};
    }
    R s, c;
    sincosR(k * Rr, &s, &c);
    return CX<R>{c * inv4pi / Rr, -s * inv4pi / Rr};
}

// Int_f 1/R dS' (s0) and Int_f R dS' (sR) over the flat triangle P at r, from the
// edge quantities of the potential integrals (Graglia 1993): per edge the
// signed in-plane distance t, the end coordinates l-, l+ and distances R-, R+;
// sR follows from div_s((rho' - rho) R) = 3R - d^2/R.
template <class R> __device__ void tri_s0_sR(const R P[3][3], const R r[3], R &s0, R &sR)
{
    const R e1[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
    const R e2[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
    R n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    const R nn = sqrtR(dot(n, n));
    n[0] /= nn; n[1] /= nn; n[2] /= nn;
    const R rp[3] = {r[0] - P[0][0], r[1] - P[0][1], r[2] - P[0][2]};
    const R dd = dot(n, rp);
    const R ad = absR(dd);
    const R rho[3] = {r[0] - dd * n[0], r[1] - dd * n[1], r[2] - dd * n[2]};
    R acc0 = 0, edgeR = 0;
    for (int e = 0; e < 3; ++e) {
        const R *a = P[e], *b = P[(e + 1) % 3];
        const R lv[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
        const R ll = sqrtR(dot(lv, lv));
        const R lh[3] = {lv[0] / ll, lv[1] / ll, lv[2] / ll};
        const R uh[3] = {lh[1] * n[2] - lh[2] * n[1], lh[2] * n[0] - lh[0] * n[2], lh[0] * n[1] - lh[1] * n[0]};
        const R am[3] = {a[0] - rho[0], a[1] - rho[1], a[2] - rho[2]};
        const R bm[3] = {b[0] - rho[0], b[1] - rho[1], b[2] - rho[2]};
        const R lp = dot(bm, lh), lm = dot(am, lh), t = dot(am, uh);
        const R R02 = t * t + dd * dd;
        const R Rp = sqrtR(R02 + lp * lp), Rm = sqrtR(R02 + lm * lm);
        R f = 0;
        if (R02 > 0) {
            f = (lm < 0 && lp < 0) ? logR((Rm - lm) / (Rp - lp)) : logR((Rp + lp) / (Rm + lm));
            R term = t * f;
            if (ad > 0) term -= ad * (atanR(t * lp / (R02 + ad * Rp)) - atanR(t * lm / (R02 + ad * Rm)));
            acc0 += term;
        }
        const R gg = (R)0.5 * ((R02 > 0 ? R02 * f : (R)0) + lp * Rp - lm * Rm);
        edgeR += t * gg;
    }
    s0 = acc0;
    sR = (dd * dd * acc0 + edgeR) / (R)3;
}

template <class R> __device__ void face_local(const VGeo &g, int f, const double *o, R P[3][3])
{
    for (int a = 0; a < 3; ++a) loc<R>(g.vtx + 3 * g.fv[3 * f + a], o, P[a]);
}

// Int_T 1/R dV' (s0v) and Int_T (r' - r)/R dV' (s1v) for tetrahedron t at r
template <class R> __device__ void tet_integrals(const VGeo &g, int t, const double *o, const R r[3], R &s0v, R s1v[3])
{
    R P[4][3];
    for (int a = 0; a < 4; ++a) loc<R>(g.vtx + 3 * g.tet[4 * t + a], o, P[a]);
    s0v = 0;
    s1v[0] = s1v[1] = s1v[2] = 0;
    for (int op = 0; op < 4; ++op) {
        R F[3][3];
        int q = 0;
        for (int a = 0; a < 4; ++a)
            if (a != op) {
                F[q][0] = P[a][0]; F[q][1] = P[a][1]; F[q][2] = P[a][2];
                ++q;
            }
        const R e1[3] = {F[1][0] - F[0][0], F[1][1] - F[0][1], F[1][2] - F[0][2]};
        const R e2[3] = {F[2][0] - F[0][0], F[2][1] - F[0][1], F[2][2] - F[0][2]};
        R n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        const R nn = sqrtR(dot(n, n));
        n[0] /= nn; n[1] /= nn; n[2] /= nn;
        const R po[3] = {P[op][0] - F[0][0], P[op][1] - F[0][1], P[op][2] - F[0][2]};
        if (dot(n, po) > 0) { n[0] = -n[0]; n[1] = -n[1]; n[2] = -n[2]; }   // outward
        R s0, sR;
        tri_s0_sR<R>(F, r, s0, sR);
        const R pr[3] = {F[0][0] - r[0], F[0][1] - r[1], F[0][2] - r[2]};
        s0v += (R)0.5 * dot(pr, n) * s0;
        s1v[0] += n[0] * sR;
        s1v[1] += n[1] * sR;
        s1v[2] += n[2] * sR;
    }
}

// I = Int_T Int_T' (r - vm).(r' - vn) G,  J = Int_T Int_T' G  (T outer, T' inner)
template <class R>
__device__ void volvol(const VGeo &g, int t, int vmi, int tp, int vni, const double *o, CX<R> &I, CX<R> &J)
{
    const R k = (R)g.k;
    const bool ex = near_pair(g.tcen + 3 * t, g.thmax[t], g.tcen + 3 * tp, g.thmax[tp]);
    R vm[3], vn[3], qj[NQT][3];
    loc<R>(g.vtx + 3 * vmi, o, vm);
    loc<R>(g.vtx + 3 * vni, o, vn);
    for (int j = 0; j < NQT; ++j) loc<R>(g.tqp + ((int64_t)tp * NQT + j) * 3, o, qj[j]);
    const R Vt = (R)g.tvol[t], Vtp = (R)g.tvol[tp];
    I = CX<R>{0, 0};
    J = CX<R>{0, 0};
    for (int i = 0; i < NQT; ++i) {
        R ri[3];
        loc<R>(g.tqp + ((int64_t)t * NQT + i) * 3, o, ri);
        const R a[3] = {ri[0] - vm[0], ri[1] - vm[1], ri[2] - vm[2]};
        CX<R> Ii{0, 0}, Ji{0, 0};
        for (int j = 0; j < NQT; ++j) {
            const R bj[3] = {qj[j][0] - vn[0], qj[j][1] - vn[1], qj[j][2] - vn[2]};
            const R dr[3] = {ri[0] - qj[j][0], ri[1] - qj[j][1], ri[2] - qj[j][2]};
            const CX<R> G = green<R>(k, sqrtR(dot(dr, dr)), ex);
            const R w = (R)0.25 * dot(a, bj);
            Ii.re += w * G.re; Ii.im += w * G.im;
            Ji.re += (R)0.25 * G.re; Ji.im += (R)0.25 * G.im;
        }
        Ii.re *= Vtp; Ii.im *= Vtp; Ji.re *= Vtp; Ji.im *= Vtp;
        if (ex) {   // analytic 1/R part in FP64 (see the note on precision above)
            double rd[3], vmd[3], vnd[3], s0v, s1v[3];
            loc<double>(g.tqp + ((int64_t)t * NQT + i) * 3, o, rd);
            loc<double>(g.vtx + 3 * vmi, o, vmd);
            loc<double>(g.vtx + 3 * vni, o, vnd);
            tet_integrals<double>(g, tp, o, rd, s0v, s1v);
            const double ad[3] = {rd[0] - vmd[0], rd[1] - vmd[1], rd[2] - vmd[2]};
            const double v1[3] = {s1v[0] + (rd[0] - vnd[0]) * s0v, s1v[1] + (rd[1] - vnd[1]) * s0v,
                                  s1v[2] + (rd[2] - vnd[2]) * s0v};
            Ii.re += (R)(dot(ad, v1) * INV4PI);
            Ji.re += (R)(s0v * INV4PI);
        }
        I.re += (R)0.25 * Ii.re; I.im += (R)0.25 * Ii.im;
        J.re += (R)0.25 * Ji.re; J.im += (R)0.25 * Ji.im;
    }
    I.re *= Vt; I.im *= Vt; J.re *= Vt; J.im *= Vt;
}

// Int_T Int_f G dS' dV  (tetrahedron t outer, face f inner)
template <class R> __device__ CX<R> volface(const VGeo &g, int t, int f, const double *o)
{
    const R k = (R)g.k;
    const bool ex = near_pair(g.tcen + 3 * t, g.thmax[t], g.fcen + 3 * f, g.fhmax[f]);
    double P[3][3];
    if (ex) face_local<double>(g, f, o, P);
    CX<R> K{0, 0};
    for (int i = 0; i < NQT; ++i) {
        R ri[3];
        loc<R>(g.tqp + ((int64_t)t * NQT + i) * 3, o, ri);
        CX<R> Ki{0, 0};
        for (int j = 0; j < NQF; ++j) {
            R rj[3];
            loc<R>(g.fqp + ((int64_t)f * NQF + j) * 3, o, rj);
            const R dr[3] = {ri[0] - rj[0], ri[1] - rj[1], ri[2] - rj[2]};
            const CX<R> G = green<R>(k, sqrtR(dot(dr, dr)), ex);
            const R w = (R)c_fw[j];
            Ki.re += w * G.re; Ki.im += w * G.im;
        }
        const R A = (R)g.farea[f];
        Ki.re *= A; Ki.im *= A;
        if (ex) {
            double rd[3], s0, sR;
            loc<double>(g.tqp + ((int64_t)t * NQT + i) * 3, o, rd);
            tri_s0_sR<double>(P, rd, s0, sR);
            Ki.re += (R)(s0 * INV4PI);
        }
        K.re += (R)0.25 * Ki.re; K.im += (R)0.25 * Ki.im;
    }
    const R Vt = (R)g.tvol[t];
    K.re *= Vt; K.im *= Vt;
    return K;
}

// Int_f Int_f' G dS' dS  (f outer, f' inner)
template <class R> __device__ CX<R> faceface(const VGeo &g, int f, int fp, const double *o)
{
    const R k = (R)g.k;
    const bool ex = near_pair(g.fcen + 3 * f, g.fhmax[f], g.fcen + 3 * fp, g.fhmax[fp]);
    double P[3][3];
    if (ex) face_local<double>(g, fp, o, P);
    CX<R> L{0, 0};
    for (int i = 0; i < NQF; ++i) {
        R ri[3];
        loc<R>(g.fqp + ((int64_t)f * NQF + i) * 3, o, ri);
        CX<R> Li{0, 0};
        for (int j = 0; j < NQF; ++j) {
            R rj[3];
            loc<R>(g.fqp + ((int64_t)fp * NQF + j) * 3, o, rj);
            const R dr[3] = {ri[0] - rj[0], ri[1] - rj[1], ri[2] - rj[2]};
            const CX<R> G = green<R>(k, sqrtR(dot(dr, dr)), ex);
            const R w = (R)c_fw[j];
            Li.re += w * G.re; Li.im += w * G.im;
        }
        const R A = (R)g.farea[fp];
        Li.re *= A; Li.im *= A;
        if (ex) {
            double rd[3], s0, sR;
            loc<double>(g.fqp + ((int64_t)f * NQF + i) * 3, o, rd);
            tri_s0_sR<double>(P, rd, s0, sR);
            Li.re += (R)(s0 * INV4PI);
        }
        const R w = (R)c_fw[i];
        L.re += w * Li.re; L.im += w * Li.im;
    }
    const R A = (R)g.farea[f];
    L.re *= A; L.im *= A;
    return L;
}

template <class R> __device__ CX<R> VGeo::entry(int m, int n) const
{
    const VGeo &g = *this;
    const double *o = g.vtx + 3 * g.fv[3 * n];
    const double k2 = g.k * g.k;
    const double qs_m = g.fqs[m], qs_n = g.fqs[n];
    CX<R> z{0, 0};
    for (int p = 0; p < 2; ++p) {
        const int t = g.ftet[2 * m + p];
        if (t < 0) continue;
        const double s = p == 0 ? 1.0 : -1.0;
        const int vm = g.ffree[2 * m + p];
        const double cm = s * g.farea[m] / (3.0 * g.tvol[t]);
        const double qm = -g.kappa[t] * s * g.farea[m] / g.tvol[t];
        for (int q = 0; q < 2; ++q) {
            const int tp = g.ftet[2 * n + q];
            if (tp < 0) continue;
            const double sp = q == 0 ? 1.0 : -1.0;
            const int vn = g.ffree[2 * n + q];
            const double cn = sp * g.farea[n] / (3.0 * g.tvol[tp]);
            const double qn = -g.kappa[tp] * sp * g.farea[n] / g.tvol[tp];
            if (t == tp) {   // Int (kappa/eps_r) f_m . f_n dV: degree 2, exact with the 4-point rule
                R vmr[3], vnr[3];
                loc<R>(g.vtx + 3 * vm, o, vmr);
                loc<R>(g.vtx + 3 * vn, o, vnr);
                R acc = 0;
                for (int i = 0; i < NQT; ++i) {
                    R ri[3];
                    loc<R>(g.tqp + ((int64_t)t * NQT + i) * 3, o, ri);
                    const R a[3] = {ri[0] - vmr[0], ri[1] - vmr[1], ri[2] - vmr[2]};
                    const R b[3] = {ri[0] - vnr[0], ri[1] - vnr[1], ri[2] - vnr[2]};
                    acc += (R)0.25 * dot(a, b);
                }
                z.re += (R)(g.kappa[t] / g.epsr[t] * cm * cn * g.tvol[t]) * acc;
            }
            CX<R> I, J;
            volvol<R>(g, t, vm, tp, vn, o, I, J);
            const R ca = (R)(-k2 * g.kappa[t] * g.kappa[tp] * cm * cn), cb = (R)(qm * qn);
            z.re += ca * I.re + cb * J.re;
            z.im += ca * I.im + cb * J.im;
        }
        if (qs_n != 0.0) {
            const CX<R> K = volface<R>(g, t, n, o);
            const R c = (R)(qm * qs_n);
            z.re += c * K.re;
            z.im += c * K.im;
        }
    }
    if (qs_m != 0.0) {
        for (int q = 0; q < 2; ++q) {
            const int tp = g.ftet[2 * n + q];
            if (tp < 0) continue;
            const double sp = q == 0 ? 1.0 : -1.0;
            const double qn = -g.kappa[tp] * sp * g.farea[n] / g.tvol[tp];
            const CX<R> K = volface<R>(g, tp, m, o);   // = Int_{face m} Int_{tp} G
            const R c = (R)(qs_m * qn);
            z.re += c * K.re;
            z.im += c * K.im;
        }
        if (qs_n != 0.0) {
            const CX<R> L = faceface<R>(g, m, n, o);
            const R c = (R)(qs_m * qs_n);
            z.re += c * L.re;
            z.im += c * L.im;
        }
    }
    return z;
}

// ---- near fill by blocks ------------------------------------------------------------
//
// The 4 + 4 + 1 element integrals of an entry (tetrahedron pairs, tetrahedron-face pairs, face
// pair) hang on the elements, and an element belongs to several of the block's functions: a
// chunk of 32 x 32 faces has about 32 tetrahedra a side, so each tetrahedron pair serves four
// to five entries and each tetrahedron-face pair two.  A CTA takes one such chunk, evaluates each
// pair once (phase 1: quadrature values of G and, for close pairs, the FP64 analytic parts at
// the four outer points) and then forms the entries from them (phase 2).
//
// The FP64 analytic parts bound it (FP64 runs at 1/64 of the FP32 rate here).  Over a
// tetrahedron at one point they take 4 vertex distances, 6 edge logarithms (an edge's logarithm
// is the same in both of its faces) and 4 arc tangents (the sum over a face's edges is the
// solid angle of the face: Van Oosterom & Strackee 1983), with all directions and normals from
// a table, where the entry function evaluates each face by itself from its vertices (24 distances,
// 12 logarithms, 24 arc tangents and 48 square roots and quotients for the directions).
// 2,808 unknowns (6^3 voxels, leaves of 44): 60 ms; one thread per entry with its own element
// integrals took 400 ms.
constexpr int FB = 32;                    // faces of a chunk side
constexpr int FG = 4;                     // inner tetrahedra per round

struct SwgJob { int64_t out; int32_t r0, c0, m, n, ld, pad; };

__device__ __forceinline__ void diff_points(const float2 *a, const float2 *b, float (&d)[3])
{
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        const float s = __fsub_rn(a[x].x, b[x].x), bb = __fsub_rn(s, a[x].x);
        const float e = __fsub_rn(__fsub_rn(a[x].x, __fsub_rn(s, bb)), __fadd_rn(b[x].x, bb));
        d[x] = __fadd_rn(s, __fadd_rn(e, __fsub_rn(a[x].y, b[x].y)));
    }
}

__device__ __forceinline__ double edge_log(double lm, double lp, double Rm, double Rp)
{
    return (lm < 0 && lp < 0) ? log((Rm - lm) / (Rp - lp)) : log((Rp + lp) / (Rm + lm));
}
__device__ __forceinline__ double dot3(const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

// |d| times the solid angle of a triangle with vertices v0, v1, v2 relative to the point (lengths R),
// d = distance of its plane, a2 = twice its area (|det(v0, v1, v2)| = a2 |d|)
__device__ __forceinline__ double plane_angle(double d, double a2, const double *v0, const double *v1, const double *v2,
                                              double R0, double R1, double R2)
{
    const double ad = fabs(d);
    if (!(ad > 0)) return 0.0;
    const double den = R0 * R1 * R2 + dot3(v0, v1) * R2 + dot3(v0, v2) * R1 + dot3(v1, v2) * R0;
    return ad * 2.0 * atan2(a2 * ad, den);
}

// Int_f 1/R dS' over face f at r
__device__ double face_s0(const double *__restrict__ F, const double *r)
{
    double v[3][3], R[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int x = 0; x < 3; ++x) v[a][x] = F[3 * a + x] - r[x];
        R[a] = sqrt(dot3(v[a], v[a]));
    }
    const double d = dot3(v[0], F + 9);
    double s0 = 0.0;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int b = (e + 1) % 3;
        const double t = dot3(v[e], F + 21 + 3 * e);
        if (t * t + d * d > 0) s0 += t * edge_log(dot3(v[e], F + 12 + 3 * e), dot3(v[b], F + 12 + 3 * e), R[e], R[b]);
    }
    return s0 - plane_angle(d, F[30], v[0], v[1], v[2], R[0], R[1], R[2]);
}

// faces of a tetrahedron (opposite vertex a): their vertices; edges 01 02 03 12 13 23 by vertex pair
__device__ constexpr int TFV[4][3] = {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}};
__device__ constexpr int TEV[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
// the edges of face a in the order (v0 v1), (v1 v2), (v0 v2)
__device__ constexpr int TFE[4][3] = {{3, 5, 4}, {1, 5, 2}, {0, 4, 2}, {0, 3, 1}};

// Int_T 1/R dV' (out[0]) and Int_T (r' - r)/R dV' (out[1..3])
__device__ void tet_s0_s1(const double *__restrict__ G, const double *r, double *out)
{
    double v[4][3], R[4], f[6], g[6];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int x = 0; x < 3; ++x) v[a][x] = G[3 * a + x] - r[x];
        R[a] = sqrt(dot3(v[a], v[a]));
    }
    const double *E = G + 12 + 4 * 13;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const int a = TEV[e][0], b = TEV[e][1];
        const double lm = dot3(v[a], E + 4 * e), lp = lm + E[4 * e + 3];
        f[e] = edge_log(lm, lp, R[a], R[b]);
        g[e] = lp * R[b] - lm * R[a];
    }
    double s0v = 0, s1[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const double *F = G + 12 + 13 * a;
        const double d = dot3(v[TFV[a][0]], F);
        double s0 = 0, eR = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int e = TFE[a][q];
            const double t = dot3(v[TEV[e][0]], F + 3 + 3 * q), r02 = t * t + d * d;
            if (r02 > 0) {
                s0 += t * f[e];
                eR += t * 0.5 * (r02 * f[e] + g[e]);
            } else {
                eR += t * 0.5 * g[e];
            }
        }
        s0 -= plane_angle(d, F[12], v[TFV[a][0]], v[TFV[a][1]], v[TFV[a][2]], R[TFV[a][0]], R[TFV[a][1]], R[TFV[a][2]]);
        const double sR = (d * d * s0 + eR) / 3.0;
        s0v += 0.5 * d * s0;
#pragma unroll
        for (int x = 0; x < 3; ++x) s1[x] += F[x] * sR;
    }
    out[0] = s0v;
    out[1] = s1[0];
    out[2] = s1[1];
    out[3] = s1[2];
}

struct SwgSide {                          // one side (rows or columns) of a chunk
    int face[FB];
    int tl[FB][2], tf[FB][2];             // local tetrahedron and free vertex of each half (-1: none)
    int tet[2 * FB], nt;
    double cm[FB][2], qm[FB][2], qs[FB];  // s a / 3V kappa and -kappa s a / V of the halves; face charge
    float pt[FB][2][NQT][3];              // quadrature points relative to the half's free vertex
};
struct SwgSmem {
    SwgSide r, c;
    int ex[2 * FB * FG];
    union {
        struct {                          // phase 1 and 2, one round
            double an[2 * FB * FG][NQT][4];   // analytic parts of (outer tetrahedron, inner of the round) at the outer points
            float2 G[2 * FB * FG][NQT][NQT];
        } v;
        double2 k[2][2 * FB][FB];         // Int_t Int_f G: row tetrahedra x column faces, column tetrahedra x row faces
    };
};

__device__ void load_side(SwgSide &S, const VGeo &g, int p0, int n)
{
    const int tid = threadIdx.x;
    if (tid < FB) S.face[tid] = tid < n ? g.perm[p0 + tid] : -1;
    __syncthreads();
    if (tid < 2 * FB) {
        const int i = tid >> 1, p = tid & 1, f = S.face[i];
        const int t = f >= 0 ? g.ftet[2 * f + p] : -1;
        S.tf[i][p] = t >= 0 ? g.ffree[2 * f + p] : -1;
        S.tl[i][p] = t;                   // the tetrahedron for now
        const double s = p == 0 ? 1.0 : -1.0;
        S.cm[i][p] = t >= 0 ? g.kappa[t] * (s * g.farea[f] / (3.0 * g.tvol[t])) : 0.0;
        S.qm[i][p] = t >= 0 ? -g.kappa[t] * s * g.farea[f] / g.tvol[t] : 0.0;
        if (p == 0) S.qs[i] = f >= 0 ? g.fqs[f] : 0.0;
    }
    __syncthreads();
    // local numbers: a half is first if no earlier half has its tetrahedron
    int mine = -1, first = -1, rank = 0;
    if (tid < 2 * FB) {
        mine = S.tl[tid >> 1][tid & 1];
        for (int k = 0; k < tid && mine >= 0; ++k)
            if (S.tl[k >> 1][k & 1] == mine) { first = k; break; }
        if (mine >= 0 && first < 0) first = tid;
    }
    __syncthreads();
    __shared__ int isf[2 * FB];
    if (tid < 2 * FB) isf[tid] = mine >= 0 && first == tid;
    __syncthreads();
    if (tid < 2 * FB && mine >= 0) {
        for (int k = 0; k < first; ++k) rank += isf[k];
        S.tl[tid >> 1][tid & 1] = rank;
        if (first == tid) S.tet[rank] = mine;
    }
    if (tid == 0) {
        int k = 0;
        for (int q = 0; q < 2 * FB; ++q) k += isf[q];
        S.nt = k;
    }
    __syncthreads();
    for (int e = tid; e < 2 * FB * NQT; e += blockDim.x) {
        const int i = e / (2 * NQT), p = e / NQT % 2, q = e % NQT;
        if (S.tl[i][p] < 0) continue;
        diff_points(g.tqp32 + 3 * ((int64_t)S.tet[S.tl[i][p]] * NQT + q), g.vtx32 + 3 * (int64_t)S.tf[i][p], S.pt[i][p][q]);
    }
    __syncthreads();
}

// Int_t Int_f G, outer point i of the four: the quad's lanes (i = lane % 4) each one point, summed
// in point order (the analytic parts in FP64)
__device__ double2 volface_quad(const VGeo &g, int t, int f, int i, float k)
{
    const bool ex = near_pair(g.tcen + 3 * (int64_t)t, g.thmax[t], g.fcen + 3 * (int64_t)f, g.fhmax[f]);
    CX<float> K{0, 0};
    for (int j = 0; j < NQF; ++j) {
        float dr[3];
        diff_points(g.tqp32 + 3 * ((int64_t)t * NQT + i), g.fqp32 + 3 * ((int64_t)f * NQF + j), dr);
        const CX<float> G = green<float>(k, sqrtf(dot(dr, dr)), ex);
        const float w = (float)c_fw[j];
        K.re += w * G.re;
        K.im += w * G.im;
    }
    double s0 = 0.0;
    if (ex) s0 = face_s0(g.fgeo + (int64_t)f * FGEO, g.tqp + 3 * ((int64_t)t * NQT + i)) * INV4PI;
    const int base = (threadIdx.x & 31) & ~3;
    float re = 0.f, im = 0.f;
    double an = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        re += 0.25f * __shfl_sync(0xffffffffu, K.re, base + q);
        im += 0.25f * __shfl_sync(0xffffffffu, K.im, base + q);
        an += 0.25 * __shfl_sync(0xffffffffu, s0, base + q);
    }
    const double V = g.tvol[t], A = g.farea[f];
    return make_double2(V * (A * re + an), V * A * im);
}

__global__ void __launch_bounds__(256)
k_fill_swg(VGeo g, const SwgJob *__restrict__ jobs, float2 *pool)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    SwgSmem &S = *reinterpret_cast<SwgSmem *>(smraw);
    const SwgJob J = jobs[blockIdx.x];
    const int tid = threadIdx.x;
    const float k = (float)g.k;
    const double k2 = g.k * g.k;
    load_side(S.r, g, J.r0, J.m);
    load_side(S.c, g, J.c0, J.n);
    const int n = tid % FB, m0 = tid / FB;         // the thread's entries: column n, rows m0 + 8 e
    // the entries in FP64: their element integrals cancel like the charges of a dipole
    double2 z[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) z[e] = make_double2(0.0, 0.0);
    const int nr = S.r.nt, nc = S.c.nt;
    for (int b0 = 0; b0 < nc; b0 += FG) {
        const int nb = min(FG, nc - b0);
        // phase 1: outer tetrahedron a, inner b0 + b, outer point i
        for (int q = tid; q < nr * nb * NQT; q += blockDim.x) {
            const int i = q % NQT, a = q / NQT % nr, b = q / (NQT * nr);
            const int t = S.r.tet[a], tp = S.c.tet[b0 + b];
            const bool ex = near_pair(g.tcen + 3 * (int64_t)t, g.thmax[t], g.tcen + 3 * (int64_t)tp, g.thmax[tp]);
            const int at = b * nr + a;
            for (int j = 0; j < NQT; ++j) {
                float dr[3];
                diff_points(g.tqp32 + 3 * ((int64_t)t * NQT + i), g.tqp32 + 3 * ((int64_t)tp * NQT + j), dr);
                const CX<float> G = green<float>(k, sqrtf(dot(dr, dr)), ex);
                S.v.G[at][i][j] = make_float2(G.re, G.im);
            }
            if (ex) tet_s0_s1(g.tgeo + (int64_t)tp * TGEO, g.tqp + 3 * ((int64_t)t * NQT + i), S.v.an[at][i]);
            if (i == 0) S.ex[at] = ex;
        }
        __syncthreads();
        // phase 2
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = m0 + 8 * e;
            if (m >= J.m || n >= J.n) continue;
            for (int q = 0; q < 2; ++q) {
                const int bl = S.c.tl[n][q] - b0;
                if (S.c.tl[n][q] < 0 || bl < 0 || bl >= nb) continue;
                const int tp = S.c.tet[b0 + bl];
                const double *vn = g.vtx + 3 * (int64_t)S.c.tf[n][q];
                for (int p = 0; p < 2; ++p) {
                    const int al = S.r.tl[m][p];
                    if (al < 0) continue;
                    const int t = S.r.tet[al], at = bl * nr + al;
                    const bool ex = S.ex[at];
                    CX<float> I{0, 0}, Jc{0, 0};
                    double aI = 0.0, aJ = 0.0;         // the analytic parts
                    for (int i = 0; i < NQT; ++i) {
                        const float *a = S.r.pt[m][p][i];
                        CX<float> Ii{0, 0}, Ji{0, 0};
#pragma unroll
                        for (int j = 0; j < NQT; ++j) {
                            const float2 G = S.v.G[at][i][j];
                            const float *b = S.c.pt[n][q][j];
                            const float w = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
                            Ii.re += w * G.x; Ii.im += w * G.y;
                            Ji.re += G.x; Ji.im += G.y;
                        }
                        I.re += Ii.re; I.im += Ii.im;
                        Jc.re += Ji.re; Jc.im += Ji.im;
                        if (ex) {
                            const double *rd = g.tqp + 3 * ((int64_t)t * NQT + i), *vm = g.vtx + 3 * (int64_t)S.r.tf[m][p];
                            const double *an = S.v.an[at][i];
#pragma unroll
                            for (int x = 0; x < 3; ++x) aI += (rd[x] - vm[x]) * (an[1 + x] + (rd[x] - vn[x]) * an[0]);
                            aJ += an[0];
                        }
                    }
                    // weights 1/4 of each point; times the volumes (the analytic parts hold the inner one)
                    const double Vt = g.tvol[t], W = Vt * g.tvol[tp] * 0.0625, Wa = Vt * 0.25 * INV4PI;
                    const double ca = -k2 * S.r.cm[m][p] * S.c.cm[n][q], cb = S.r.qm[m][p] * S.c.qm[n][q];
                    z[e].x += ca * (W * I.re + Wa * aI) + cb * (W * Jc.re + Wa * aJ);
                    z[e].y += W * (ca * I.im + cb * Jc.im);
                    if (t == tp && g.kappa[t] != 0.0) {   // Int (kappa/eps_r) f_m . f_n dV: degree 2, exact with the 4-point rule
                        float acc = 0.f;
                        for (int i = 0; i < NQT; ++i) {
                            const float *a = S.r.pt[m][p][i], *b = S.c.pt[n][q][i];
                            acc += 0.25f * (a[0] * b[0] + a[1] * b[1] + a[2] * b[2]);
                        }
                        z[e].x += S.r.cm[m][p] * S.c.cm[n][q] * g.tvol[t] / (g.kappa[t] * g.epsr[t]) * acc;
                    }
                }
            }
        }
        __syncthreads();
    }
    // tetrahedron-face integrals, both ways (a quad of lanes each; all lanes run the same rounds)
    for (int side = 0; side < 2; ++side) {
        const SwgSide &T = side ? S.c : S.r, &F = side ? S.r : S.c;
        const int nf = side ? J.m : J.n, total = T.nt * nf;
        for (int q0 = 0; q0 < total; q0 += blockDim.x / 4) {
            const int q = min(q0 + tid / 4, total - 1), a = q / nf, f = q % nf;
            const double2 K = volface_quad(g, T.tet[a], F.face[f], tid & 3, k);
            if ((tid & 3) == 0) S.k[side][a][f] = K;
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int m = m0 + 8 * e;
        if (m >= J.m || n >= J.n) continue;
        const double qsm = S.r.qs[m], qsn = S.c.qs[n];
        for (int p = 0; p < 2; ++p) {
            const int al = S.r.tl[m][p], bl = S.c.tl[n][p];
            if (qsn != 0.0 && al >= 0) {
                const double2 K = S.k[0][al][n];
                const double c = S.r.qm[m][p] * qsn;
                z[e].x += c * K.x;
                z[e].y += c * K.y;
            }
            if (qsm != 0.0 && bl >= 0) {
                const double2 K = S.k[1][bl][m];
                const double c = qsm * S.c.qm[n][p];
                z[e].x += c * K.x;
                z[e].y += c * K.y;
            }
        }
        if (qsm != 0.0 && qsn != 0.0) {     // Int_m Int_n G
            const int f = S.r.face[m], fp = S.c.face[n];
            const bool ex = near_pair(g.fcen + 3 * (int64_t)f, g.fhmax[f], g.fcen + 3 * (int64_t)fp, g.fhmax[fp]);
            CX<float> L{0, 0};
            double an = 0.0;
            for (int i = 0; i < NQF; ++i) {
                CX<float> Li{0, 0};
                for (int j = 0; j < NQF; ++j) {
                    float dr[3];
                    diff_points(g.fqp32 + 3 * ((int64_t)f * NQF + i), g.fqp32 + 3 * ((int64_t)fp * NQF + j), dr);
                    const CX<float> G = green<float>(k, sqrtf(dot(dr, dr)), ex);
                    const float w = (float)c_fw[j];
                    Li.re += w * G.re;
                    Li.im += w * G.im;
                }
                if (ex) an += c_fw[i] * face_s0(g.fgeo + (int64_t)fp * FGEO, g.fqp + 3 * ((int64_t)f * NQF + i));
                const float w = (float)c_fw[i];
                L.re += w * Li.re;
                L.im += w * Li.im;
            }
            const double A = g.farea[f], Ap = g.farea[fp], c = qsm * qsn * A;
            z[e].x += c * (Ap * L.re + INV4PI * an);
            z[e].y += c * Ap * L.im;
        }
        pool[J.out + (int64_t)m * J.ld + n] = make_float2((float)z[e].x, (float)z[e].y);
    }
}

hm_status VGeo::fill_near(const std::vector<FillJob> &fj, float2 *pool, TmpBuffers &tmp, cudaStream_t s) const
{
    std::vector<SwgJob> jobs;
    for (const FillJob &f : fj) {         // even chunks of at most FB faces a side
        const int nm = (f.m + FB - 1) / FB, nn = (f.n + FB - 1) / FB;
        for (int a = 0; a < nm; ++a)
            for (int b = 0; b < nn; ++b) {
                const int i0 = f.m * a / nm, i1 = f.m * (a + 1) / nm, j0 = f.n * b / nn, j1 = f.n * (b + 1) / nn;
                jobs.push_back({f.out + (int64_t)i0 * f.ld + j0, f.r0 + i0, f.c0 + j0, i1 - i0, j1 - j0, f.ld, 0});
            }
    }
    if (jobs.empty()) return HM_OK;
    SwgJob *d_jobs = nullptr;
    const hm_status st = tmp.up(&d_jobs, jobs, s);
    if (st != HM_OK) return st;
    HM_CUDA(cudaFuncSetAttribute(k_fill_swg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SwgSmem)));
    k_fill_swg<<<(unsigned)jobs.size(), 256, sizeof(SwgSmem), s>>>(*this, d_jobs, pool);
    HM_CUDA(cudaGetLastError());
    return HM_OK;
}

static double norm3(const double *d) { return std::sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]); }

static double max_edge(const double *const *p, int np)
{
    double h = 0.0;
    for (int i = 0; i < np; ++i)
        for (int j = i + 1; j < np; ++j) {
            const double d[3] = {p[i][0] - p[j][0], p[i][1] - p[j][1], p[i][2] - p[j][2]};
            const double l = norm3(d);
            if (l > h) h = l;
        }
    return h;
}

} // namespace

hm_status swg_faces(int64_t nv, int64_t nt, const int32_t *tet, std::vector<int32_t> &fv, std::vector<int32_t> &ftet,
                    std::vector<int32_t> &ffree)
{
    struct HF { std::array<int32_t, 3> key; int32_t t, w; };
    std::vector<HF> hf;
    hf.reserve(4 * nt);
    for (int64_t t = 0; t < nt; ++t) {
        const int32_t *v = tet + 4 * t;
        for (int a = 0; a < 4; ++a) {
            if (v[a] < 0 || v[a] >= nv) return fail(HM_ERR_ARG, "tetrahedron vertex id out of range");
            for (int b = a + 1; b < 4; ++b)
                if (v[a] == v[b]) return fail(HM_ERR_ARG, "tetrahedron with a repeated vertex");
        }
        for (int op = 0; op < 4; ++op) {
            std::array<int32_t, 3> k{};
            int q = 0;
            for (int a = 0; a < 4; ++a)
                if (a != op) k[q++] = v[a];
            std::sort(k.begin(), k.end());
            hf.push_back({k, (int32_t)t, v[op]});
        }
    }
    std::sort(hf.begin(), hf.end(), [](const HF &x, const HF &y) { return x.key < y.key || (x.key == y.key && x.t < y.t); });
    fv.clear(); ftet.clear(); ffree.clear();
    for (size_t i = 0; i < hf.size();) {
        size_t j = i;
        while (j < hf.size() && hf[j].key == hf[i].key) ++j;
        if (j - i > 2) return fail(HM_ERR_ARG, "a face is shared by more than two tetrahedra");
        fv.insert(fv.end(), hf[i].key.begin(), hf[i].key.end());
        ftet.push_back(hf[i].t);
        ffree.push_back(hf[i].w);
        ftet.push_back(j - i == 2 ? hf[i + 1].t : -1);
        ffree.push_back(j - i == 2 ? hf[i + 1].w : -1);
        i = j;
    }
    return HM_OK;
}

hm_status build_from_tets(const hm_mesh *mesh, const hm_build_opts *o, cudaStream_t s, hm_matrix *out)
{
    const int64_t nv = mesh->n_vert, nt = mesh->n_cell;
    if (nv < 4 || nt < 1 || !mesh->xyz || !mesh->cells) return fail(HM_ERR_ARG, "empty mesh");
    if (!mesh->eps_r) return fail(HM_ERR_ARG, "eps_r is required for an SWG mesh");
    for (int64_t t = 0; t < nt; ++t)
        if (!(mesh->eps_r[t] > 0) || !std::isfinite(mesh->eps_r[t])) return fail(HM_ERR_ARG, "eps_r must be finite and > 0");
    std::vector<int32_t> fv, ftet, ffree;
    hm_status st = swg_faces(nv, nt, mesh->cells, fv, ftet, ffree);
    if (st != HM_OK) return st;
    const int64_t N = (int64_t)fv.size() / 3;
    const double *X = mesh->xyz;

    // ---- tetrahedra
    const double ta = (5.0 + 3.0 * std::sqrt(5.0)) / 20.0, tb = (5.0 - std::sqrt(5.0)) / 20.0;
    std::vector<double> tqp(3 * NQT * nt), tcen(3 * nt), thmax(nt), tvol(nt), kappa(nt), epsr(mesh->eps_r, mesh->eps_r + nt);
    for (int64_t t = 0; t < nt; ++t) {
        const double *p[4];
        for (int a = 0; a < 4; ++a) p[a] = X + 3 * mesh->cells[4 * t + a];
        const double e1[3] = {p[1][0] - p[0][0], p[1][1] - p[0][1], p[1][2] - p[0][2]};
        const double e2[3] = {p[2][0] - p[0][0], p[2][1] - p[0][1], p[2][2] - p[0][2]};
        const double e3[3] = {p[3][0] - p[0][0], p[3][1] - p[0][1], p[3][2] - p[0][2]};
        const double cr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        tvol[t] = std::fabs(cr[0] * e3[0] + cr[1] * e3[1] + cr[2] * e3[2]) / 6.0;
        if (!(tvol[t] > 0)) return fail(HM_ERR_ARG, "degenerate tetrahedron (zero volume)");
        for (int d = 0; d < 3; ++d) tcen[3 * t + d] = (p[0][d] + p[1][d] + p[2][d] + p[3][d]) / 4.0;
        thmax[t] = max_edge(p, 4);
        kappa[t] = 1.0 - 1.0 / epsr[t];
        for (int q = 0; q < NQT; ++q)
            for (int d = 0; d < 3; ++d) {
                double acc = 0.0;
                for (int a = 0; a < 4; ++a) acc = acc + (q == a ? ta : tb) * p[a][d];
                tqp[(t * NQT + q) * 3 + d] = acc;
            }
    }
    // ---- faces
    const double s15 = std::sqrt(15.0);
    const double a1 = (6.0 - s15) / 21.0, b1 = (9.0 + 2.0 * s15) / 21.0;
    const double a2 = (6.0 + s15) / 21.0, b2 = (9.0 - 2.0 * s15) / 21.0;
    const double bary[NQF][3] = {{1.0 / 3, 1.0 / 3, 1.0 / 3}, {a1, a1, b1}, {a1, b1, a1}, {b1, a1, a1},
                                 {a2, a2, b2}, {a2, b2, a2}, {b2, a2, a2}};
    const double fw[NQF] = {9.0 / 40.0, (155.0 - s15) / 1200.0, (155.0 - s15) / 1200.0, (155.0 - s15) / 1200.0,
                            (155.0 + s15) / 1200.0, (155.0 + s15) / 1200.0, (155.0 + s15) / 1200.0};
    std::vector<double> fqp(3 * NQF * N), fcen(3 * N), fhmax(N), farea(N), fqs(N);
    BasisData B;
    B.N = N;
    for (int64_t f = 0; f < N; ++f) {
        const double *p[3];
        for (int a = 0; a < 3; ++a) p[a] = X + 3 * fv[3 * f + a];
        const double e1[3] = {p[1][0] - p[0][0], p[1][1] - p[0][1], p[1][2] - p[0][2]};
        const double e2[3] = {p[2][0] - p[0][0], p[2][1] - p[0][1], p[2][2] - p[0][2]};
        const double cr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        farea[f] = 0.5 * norm3(cr);
        for (int d = 0; d < 3; ++d) fcen[3 * f + d] = (p[0][d] + p[1][d] + p[2][d]) / 3.0;
        fhmax[f] = max_edge(p, 3);
        for (int q = 0; q < NQF; ++q)
            for (int d = 0; d < 3; ++d)
                fqp[(f * NQF + q) * 3 + d] = bary[q][0] * p[0][d] + bary[q][1] * p[1][d] + bary[q][2] * p[2][d];
        const int tp = ftet[2 * f], tm = ftet[2 * f + 1];
        fqs[f] = kappa[tp] - (tm >= 0 ? kappa[tm] : 0.0);
        // tree: face centroid; support box: the vertices of T+ and T-
        for (int d = 0; d < 3; ++d) B.cen.push_back(fcen[3 * f + d]);
        const double *pp[5] = {p[0], p[1], p[2], X + 3 * ffree[2 * f], X + 3 * (tm >= 0 ? ffree[2 * f + 1] : ffree[2 * f])};
        for (int d = 0; d < 3; ++d) {
            double lo = INFINITY, hi = -INFINITY;
            for (int q = 0; q < 5; ++q) {
                lo = std::min(lo, pp[q][d]);
                hi = std::max(hi, pp[q][d]);
            }
            B.blo.push_back(lo);
            B.bhi.push_back(hi);
        }
    }
    // geometry of the analytic integrals (k_fill_swg): directions, in-plane outward normals, areas
    std::vector<double> fgeo((size_t)N * FGEO), tgeo((size_t)nt * TGEO);
    auto sub = [](const double *a, const double *b, double *o) { for (int d = 0; d < 3; ++d) o[d] = a[d] - b[d]; };
    auto unit = [](double *a) {
        const double l = norm3(a);
        for (int d = 0; d < 3; ++d) a[d] /= l;
        return l;
    };
    auto cross = [](const double *a, const double *b, double *o) {
        o[0] = a[1] * b[2] - a[2] * b[1]; o[1] = a[2] * b[0] - a[0] * b[2]; o[2] = a[0] * b[1] - a[1] * b[0];
    };
    auto dotd = [](const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
    // unit normal of the triangle (p0, p1, p2) and twice its area
    auto plane = [&](const double *p0, const double *p1, const double *p2, double *n) {
        double a[3], b[3];
        sub(p1, p0, a);
        sub(p2, p0, b);
        cross(a, b, n);
        return unit(n);
    };
    // the in-plane unit normal of the edge a b of a triangle with normal n, away from its vertex c
    auto outward = [&](const double *a, const double *b, const double *c, const double *n, double *u) {
        double l[3], w[3];
        sub(b, a, l);
        unit(l);
        cross(l, n, u);
        sub(c, a, w);
        if (dotd(u, w) > 0)
            for (int d = 0; d < 3; ++d) u[d] = -u[d];
    };
    for (int64_t f = 0; f < N; ++f) {
        double *G = &fgeo[(size_t)f * FGEO];
        const double *p[3];
        for (int a = 0; a < 3; ++a) {
            p[a] = X + 3 * fv[3 * f + a];
            for (int d = 0; d < 3; ++d) G[3 * a + d] = p[a][d];
        }
        G[30] = plane(p[0], p[1], p[2], G + 9);
        for (int e = 0; e < 3; ++e) {
            sub(p[(e + 1) % 3], p[e], G + 12 + 3 * e);
            unit(G + 12 + 3 * e);
            outward(p[e], p[(e + 1) % 3], p[(e + 2) % 3], G + 9, G + 21 + 3 * e);
        }
    }
    static const int TV[4][3] = {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}};
    static const int TE[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
    for (int64_t t = 0; t < nt; ++t) {
        double *G = &tgeo[(size_t)t * TGEO];
        const double *p[4];
        for (int a = 0; a < 4; ++a) {
            p[a] = X + 3 * mesh->cells[4 * t + a];
            for (int d = 0; d < 3; ++d) G[3 * a + d] = p[a][d];
        }
        for (int a = 0; a < 4; ++a) {
            const double *v0 = p[TV[a][0]], *v1 = p[TV[a][1]], *v2 = p[TV[a][2]];
            double *F = G + 12 + 13 * a, w[3];
            F[12] = plane(v0, v1, v2, F);
            sub(p[a], v0, w);
            if (dotd(F, w) > 0)
                for (int d = 0; d < 3; ++d) F[d] = -F[d];
            outward(v0, v1, v2, F, F + 3);
            outward(v1, v2, v0, F, F + 6);
            outward(v0, v2, v1, F, F + 9);
        }
        for (int e = 0; e < 6; ++e) {
            double *E = G + 12 + 52 + 4 * e;
            sub(p[TE[e][1]], p[TE[e][0]], E);
            E[3] = unit(E);
        }
    }
    HM_CUDA(cudaMemcpyToSymbol(c_fw, fw, sizeof(fw)));
    TmpBuffers tmp;
    std::vector<double> vtx(X, X + 3 * nv);
    std::vector<int32_t> tetv(mesh->cells, mesh->cells + 4 * nt);
    VGeo g{};
    double *d_vtx, *d_tqp, *d_tcen, *d_thmax, *d_tvol, *d_kappa, *d_epsr, *d_fqp, *d_fcen, *d_fhmax, *d_farea, *d_fqs;
    int32_t *d_tet, *d_fv, *d_ftet, *d_ffree;
    if ((st = tmp.up(&d_vtx, vtx, s)) || (st = tmp.up(&d_tet, tetv, s)) || (st = tmp.up(&d_tqp, tqp, s)) ||
        (st = tmp.up(&d_tcen, tcen, s)) || (st = tmp.up(&d_thmax, thmax, s)) || (st = tmp.up(&d_tvol, tvol, s)) ||
        (st = tmp.up(&d_kappa, kappa, s)) || (st = tmp.up(&d_epsr, epsr, s)) || (st = tmp.up(&d_fv, fv, s)) ||
        (st = tmp.up(&d_ftet, ftet, s)) || (st = tmp.up(&d_ffree, ffree, s)) || (st = tmp.up(&d_fqp, fqp, s)) ||
        (st = tmp.up(&d_fcen, fcen, s)) || (st = tmp.up(&d_fhmax, fhmax, s)) || (st = tmp.up(&d_farea, farea, s)) ||
        (st = tmp.up(&d_fqs, fqs, s)))
        return st;
    g.vtx = d_vtx; g.tet = d_tet; g.tqp = d_tqp; g.tcen = d_tcen; g.thmax = d_thmax; g.tvol = d_tvol;
    g.kappa = d_kappa; g.epsr = d_epsr; g.fv = d_fv; g.ftet = d_ftet; g.ffree = d_ffree; g.fqp = d_fqp;
    g.fcen = d_fcen; g.fhmax = d_fhmax; g.farea = d_farea; g.fqs = d_fqs;
    g.k = 2.0 * 3.14159265358979323846 / mesh->wavelength;
    float2 *d_vtx32, *d_tqp32, *d_fqp32;
    double *d_fgeo, *d_tgeo;
    const std::array<double, 3> mid = middle(vtx);
    if ((st = tmp.up(&d_vtx32, float_pairs(vtx, mid), s)) || (st = tmp.up(&d_tqp32, float_pairs(tqp, mid), s)) ||
        (st = tmp.up(&d_fqp32, float_pairs(fqp, mid), s)) || (st = tmp.up(&d_fgeo, fgeo, s)) || (st = tmp.up(&d_tgeo, tgeo, s)))
        return st;
    g.vtx32 = d_vtx32; g.tqp32 = d_tqp32; g.fqp32 = d_fqp32; g.fgeo = d_fgeo; g.tgeo = d_tgeo;

    // excitation: b_m = sum_s (s kappa_s a / 3) sum_q (1/4) (r_q - v_s) . p exp(-jk k . r_q)
    B.nq = NQT;
    B.qw.assign(NQT, 0.25);
    B.qpd = tqp;
    B.vtx = vtx;
    B.ucell = ftet;
    B.ufree = ffree;
    B.ucoef.resize(2 * N);
    for (int64_t f = 0; f < N; ++f)
        for (int p = 0; p < 2; ++p) {
            const int t = ftet[2 * f + p];
            B.ucoef[2 * f + p] = t < 0 ? 0.0 : (p == 0 ? 1.0 : -1.0) * kappa[t] * farea[f] / 3.0;
        }
    st = assemble(B, g, o, tmp, s, out);
    if (st == HM_OK) (*out)->basis = HM_SWG;
    return st;
}

} // namespace hm
