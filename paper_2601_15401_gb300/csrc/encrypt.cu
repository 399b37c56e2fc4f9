// Steps on either side of the multiplication (Section II): public key,
// encryption and decryption, on the device.
//
//   pk = (-a s + e, a)                        a uniform (NTT domain), s, e small
//   ct = (v pk_0 + e_0 + m, v pk_1 + e_1)     v, e_0, e_1 small, m the message
//   m' = c_0 + c_1 s                          over the two lowest limbs, lifted
//                                             by CRT (Garner, exact 128-bit) and
//                                             centred, as a double
// Everything is in the NTT domain except the small signed inputs, which are
// reduced into every limb and transformed by the library's NTT.
#include <algorithm>

#include "../../include/ckks_mulk.h"
#include "engine.h"
#include "internal.h"
#include "rns.h"

using namespace ckks;


namespace {

constexpr int kThr = 256;

__device__ __forceinline__ u64 mulmod_full(u64 a, u64 b, ModQ m, u64 r2) {
    return mont_mul(mont_mul(a, b, m), r2, m);
}

// pk0 = E - a S over `limbs` limbs (prime index = limb index)
__global__ void pk_kernel(const u64 *S, const u64 *E, const u64 *a, u64 *pk, int limbs, int N, const ModQ *mods,
                          const u64 *r2) {
    const i64 gid = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    const i64 plane = (i64)limbs * N;
    if (gid >= plane) return;
    const int x = (int)(gid / N);
    const ModQ m = mods[x];
    pk[gid] = sub_mod(E[gid], mulmod_full(a[gid], S[gid], m, r2[x]), m.q);
    pk[plane + gid] = a[gid];
}

// Garner lift of (x0 mod q0, x1 mod q1) to [0, q0 q1), centred, as double.
__global__ void crt2_kernel(const u64 *P, double *out, int limbs, int N, u64 q0, u64 q1, Shoup q0inv_mod_q1,
                            Shoup one_q1) {
    grid_dependency_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    P += (i64)blockIdx.y * limbs * N;  // batch element
    out += (i64)blockIdx.y * N;
    const u64 x0 = P[i];
    if (limbs == 1) {
        out[i] = x0 > q0 / 2 ? -(double)(q0 - x0) : (double)x0;
        return;
    }
    const u64 x1 = P[N + i];
    const u64 x0r = shoup(x0, one_q1.w, one_q1.wp, q1);  // x0 mod q1
    const u64 t = shoup(sub_mod(x1, x0r, q1), q0inv_mod_q1.w, q0inv_mod_q1.wp, q1);
    // x = x0 + q0 t < q0 q1 < 2^122
    unsigned __int128 x = (unsigned __int128)q0 * t + x0;
    const unsigned __int128 Q = (unsigned __int128)q0 * q1;
    if (x > Q / 2) {
        const unsigned __int128 y = Q - x;
        out[i] = -((double)(u64)(y >> 64) * 18446744073709551616.0 + (double)(u64)y);
    } else {
        out[i] = (double)(u64)(x >> 64) * 18446744073709551616.0 + (double)(u64)x;
    }
}

// c0 = V pk0 + T, c1 = V pk1 + E1 for every batch element (blockIdx.y), with
// T the transform of e0 + m
__global__ void enc_batch_kernel(const u64 *W, const u64 *pk, i64 pk_pstride, u64 *out, i64 out_bstride,
                                 i64 out_pstride, int level, int N, const ModQ *mods, const u64 *r2) {
    grid_dependency_wait();
    const i64 gid = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (i64)level * N) return;
    const int b = blockIdx.y;
    const int x = (int)(gid / N);
    const ModQ m = mods[x];
    const u64 q = m.q;
    const i64 plane = (i64)level * N;
    const u64 *w = W + (i64)b * 3 * plane + gid;  // V, T, E1
    u64 *c0 = out + (i64)b * out_bstride + gid, *c1 = c0 + out_pstride;
    const u64 v = mont_mul(w[0], r2[x], m);  // V R, so that one REDC per product is left
    *c0 = add_mod(mont_mul(v, pk[gid], m), w[plane], q);
    *c1 = add_mod(mont_mul(v, pk[pk_pstride + gid], m), w[2 * plane], q);
}

// P[b][x] = C0 + C1 S over the lowest `limbs` limbs of every batch element
__global__ void dec_batch_kernel(const u64 *ct, i64 bstride, i64 pstride, const u64 *S, u64 *P, int limbs, int N,
                                 const ModQ *mods, const u64 *r2) {
    grid_dependency_wait();
    const i64 gid = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (i64)limbs * N) return;
    const int b = blockIdx.y;
    const int x = (int)(gid / N);
    const ModQ m = mods[x];
    const u64 *c0 = ct + (i64)b * bstride + gid;
    P[(i64)b * limbs * N + gid] = add_mod(c0[0], mulmod_full(c0[pstride], S[gid], m, r2[x]), m.q);
}

unsigned blocks(i64 n) { return (unsigned)((n + kThr - 1) / kThr); }

u64 host_inv(u64 a, u64 q) {
    unsigned __int128 r = 1, b = a % q;
    u64 e = q - 2;
    while (e) {
        if (e & 1) r = r * b % q;
        b = b * b % q;
        e >>= 1;
    }
    return (u64)r;
}

size_t enc_batch_ws(const Context &C, uint32_t level, uint32_t batch) {
    const uint32_t chunk = std::min<uint32_t>(16383u, 65535u / (4u * level));
    return (size_t)std::min(batch, chunk) * 4 * level * C.N * sizeof(u64);  // three planes are used
}

size_t dec_batch_ws(const Context &C, uint32_t batch) {
    return ((size_t)(C.L + C.K) * C.N + (size_t)batch * 2 * C.N) * sizeof(u64);
}

// evenly spaced tuple array: batch stride in elements, -1 if not
i64 spacing(const ckks_tuple *t, uint32_t batch) {
    const i64 bs = batch > 1 ? (i64)(t[1].data - t[0].data) : 0;
    for (uint32_t b = 0; b < batch; ++b)
        if (t[b].data != t[0].data + b * bs) return -1;
    return bs;
}

}  // namespace

extern "C" {

int ckks_encrypt_workspace_size(const ckks_context *ctx, size_t *bytes) {
    if (!ctx || !bytes) return CKKS_EINVAL;
    *bytes = (size_t)4 * (ctx->c.L + ctx->c.K) * ctx->c.N * sizeof(u64);
    return CKKS_OK;
}

int ckks_public_key(ckks_context *ctx, const int64_t *s, const uint64_t *a, const int64_t *e, uint64_t *pk,
                    void *workspace, size_t ws_bytes, void *stream) {
    if (!ctx || !s || !a || !e || !pk || !workspace) return CKKS_EINVAL;
    const Context &C = ctx->c;
    size_t need;
    ckks_encrypt_workspace_size(ctx, &need);
    if (ws_bytes < need) return CKKS_ENOMEM;
    cudaSetDevice(C.device);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t plane = (size_t)(C.L + C.K) * C.N;
    u64 *S = (u64 *)workspace, *E = S + plane;
    const u64 *sa[2] = {(const u64 *)s, (const u64 *)e}, *sb[2] = {nullptr, nullptr};
    cudaError_t err = transform_signed(C, 1, 2, C.L, sa, sb, LimbView{S, 0, (i64)plane}, st);
    if (err == cudaSuccess) {
        count_kernel(C);
        pk_kernel<<<blocks((i64)C.L * C.N), kThr, 0, st>>>(S, E, (const u64 *)a, (u64 *)pk, C.L, C.N, C.d_mods, C.d_r2);
        err = cudaGetLastError();
    }
    if (err != cudaSuccess) {
        const_cast<Context &>(C).sticky.store((int)err);
        return CKKS_ECUDA;
    }
    return CKKS_OK;
}

int ckks_encrypt_batch_workspace_size(const ckks_context *ctx, uint32_t level, uint32_t batch, size_t *bytes) {
    if (!ctx || !bytes || batch < 1) return CKKS_EINVAL;
    if (level < 1 || level > (uint32_t)ctx->c.L) return CKKS_ELEVEL;
    *bytes = enc_batch_ws(ctx->c, level, batch);
    return CKKS_OK;
}

int ckks_encrypt_batch(ckks_context *ctx, const int64_t *m, const int64_t *v, const int64_t *e0, const int64_t *e1,
                       uint32_t batch, const uint64_t *pk, uint32_t level, ckks_tuple *out, void *workspace,
                       size_t ws_bytes, void *stream) {
    if (!ctx || !m || !v || !e0 || !e1 || !pk || !out || !workspace || batch < 1) return CKKS_EINVAL;
    const Context &C = ctx->c;
    if (level < 1 || level > (uint32_t)C.L) return CKKS_ELEVEL;
    for (uint32_t b = 0; b < batch; ++b) {
        if (!out[b].data) return CKKS_EINVAL;
        if (out[b].poly_stride == 0) out[b].poly_stride = level;
        if (out[b].poly_stride < level || out[b].poly_stride != out[0].poly_stride) return CKKS_EINVAL;
    }
    const i64 os = spacing(out, batch);
    if (os < 0 || (batch > 1 && os == 0)) return CKKS_EINVAL;
    if (ws_bytes < enc_batch_ws(C, level, batch)) return CKKS_ENOMEM;
    cudaSetDevice(C.device);
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t chunk = std::min<uint32_t>(16383u, 65535u / (4u * level));
    const i64 N = C.N, ps = (i64)out[0].poly_stride * N;
    u64 *W = (u64 *)workspace;
    cudaError_t err = cudaSuccess;
    for (uint32_t b0 = 0; b0 < batch && err == cudaSuccess; b0 += chunk) {
        const uint32_t cb = std::min(chunk, batch - b0);
        // V = NTT(v), T = NTT(e0 + m), E1 = NTT(e1): the signed inputs are
        // reduced into every limb as the transform loads them, and e0 and m
        // take one transform together
        const u64 *sa[3] = {(const u64 *)v + b0 * N, (const u64 *)e0 + b0 * N, (const u64 *)e1 + b0 * N};
        const u64 *sb[3] = {nullptr, (const u64 *)m + b0 * N, nullptr};
        LimbView w{W, 3 * (i64)level * N, (i64)level * N};
        err = transform_signed(C, (int)cb, 3, (int)level, sa, sb, w, st);
        if (err == cudaSuccess) {
            count_kernel(C);
            err = launch_dependent(enc_batch_kernel, dim3(blocks((i64)level * N), cb), dim3(kThr), 0, st, W, (const u64 *)pk, (i64)C.L * N, (u64 *)out[b0].data, os, ps, (int)level, C.N, C.d_mods, C.d_r2);
        }
    }
    if (err != cudaSuccess) {
        const_cast<Context &>(C).sticky.store((int)err);
        return CKKS_ECUDA;
    }
    for (uint32_t b = 0; b < batch; ++b) {
        out[b].n_polys = 2;
        out[b].level = level;
        out[b].ntt_form = 1;
    }
    return CKKS_OK;
}

int ckks_encrypt(ckks_context *ctx, const int64_t *m, const int64_t *v, const int64_t *e0, const int64_t *e1,
                 const uint64_t *pk, uint32_t level, ckks_tuple *out, void *workspace, size_t ws_bytes,
                 void *stream) {
    return ckks_encrypt_batch(ctx, m, v, e0, e1, 1, pk, level, out, workspace, ws_bytes, stream);
}

int ckks_decrypt_batch_workspace_size(const ckks_context *ctx, uint32_t batch, size_t *bytes) {
    if (!ctx || !bytes || batch < 1) return CKKS_EINVAL;
    *bytes = dec_batch_ws(ctx->c, batch);
    return CKKS_OK;
}

int ckks_decrypt_batch(ckks_context *ctx, const ckks_tuple *ct, uint32_t batch, const int64_t *s, double *out,
                       void *workspace, size_t ws_bytes, void *stream) {
    if (!ctx || !ct || !s || !out || !workspace || batch < 1 || batch > 32767) return CKKS_EINVAL;
    const Context &C = ctx->c;
    for (uint32_t b = 0; b < batch; ++b) {
        if (!ct[b].data || ct[b].n_polys != 2 || !ct[b].ntt_form || ct[b].level < 1 ||
            ct[b].level > (uint32_t)C.L || ct[b].poly_stride < ct[b].level || ct[b].level != ct[0].level ||
            ct[b].poly_stride != ct[0].poly_stride)
            return CKKS_EINVAL;
    }
    const i64 cs = spacing(ct, batch);
    if (cs < 0) return CKKS_EINVAL;
    if (ws_bytes < dec_batch_ws(C, batch)) return CKKS_ENOMEM;
    cudaSetDevice(C.device);
    cudaStream_t st = (cudaStream_t)stream;
    const int limbs = ct[0].level >= 2 ? 2 : 1;
    const i64 N = C.N;
    u64 *S = (u64 *)workspace, *P = S + (size_t)(C.L + C.K) * N;
    const u64 *sa[1] = {(const u64 *)s}, *sb[1] = {nullptr};
    cudaError_t err = transform_signed(C, 1, 1, limbs, sa, sb, LimbView{S, 0, (i64)limbs * N}, st);
    if (err == cudaSuccess) {
        count_kernel(C);
        err = launch_dependent(dec_batch_kernel, dim3(blocks((i64)limbs * N), batch), dim3(kThr), 0, st, (const u64 *)ct[0].data, cs, (i64)ct[0].poly_stride * N, S, P, limbs, C.N, C.d_mods, C.d_r2);
    }
    if (err == cudaSuccess) {
        LimbView v{P, (i64)limbs * N, (i64)limbs * N};
        err = transform_plain(C, false, (int)batch, 1, limbs, v, v, st);
    }
    if (err == cudaSuccess) {
        const u64 q0 = C.primes[0], q1 = limbs > 1 ? C.primes[1] : 1;
        Shoup inv{0, 0}, one_q1{0, 0};
        if (limbs > 1) {
            inv = make_shoup(host_inv(q0 % q1, q1), q1);
            one_q1 = make_shoup(1, q1);
        }
        count_kernel(C);
        err = launch_dependent(crt2_kernel, dim3(blocks(N), batch), dim3(kThr), 0, st, P, out, limbs, C.N, q0, q1, inv, one_q1);
    }
    if (err != cudaSuccess) {
        const_cast<Context &>(C).sticky.store((int)err);
        return CKKS_ECUDA;
    }
    return CKKS_OK;
}

int ckks_decrypt(ckks_context *ctx, const ckks_tuple *ct, const int64_t *s, double *out, void *workspace,
                 size_t ws_bytes, void *stream) {
    return ckks_decrypt_batch(ctx, ct, 1, s, out, workspace, ws_bytes, stream);
}

}  // extern "C"
