// Misfit gradient with respect to the velocity model: forward shot with
// checkpoints, then a backward sweep of hand-written adjoint steps with the
// forward recomputed segment by segment.  Included at the end of seisgb.cu.
//
// Adjoint notes (the paper has no adjoint; this is the exact discrete adjoint
// of the fused step).  With lambda^k the multiplier of u^k and M the
// coefficient of (L u + phi + f) in the update (m inside, m / (1 + e) in the
// PML), the scaled multiplier w = M lambda obeys, for k = nt .. 1:
//   w^k   = 2 w^{k+1} - w^{k+2} + m (L w^{k+1} + psi + K^T r^{k-1})         inside
//   w^k   = [(2 - e^2) w^{k+1} - (1 - e) w^{k+2} + m (L w^{k+1} + psi)] / (1 + e)  PML
//   nu^k  = nu^{k+1} / (1 + e) + w^{k+1}                             PML points
//   psi   = sum_a [c_a nu^{k+1}](x + e_a) - [c_a nu^{k+1}](x - e_a),  over PML
//           neighbours, c_a / (2 h_a) = k_a (d(+1)^2 - d(-1)^2) / (1 + e)
//   dJ/dm += w^k g^{k-1} / m,   g^n = L u^n + phi^n + f^n
// i.e. the forward step run backward in time with the trace residual r
// injected at the receivers.  dJ/dv = dJ/dm * 2 v dt^2 = 2 (sum_k w^k g^{k-1}) / v
// (dt held fixed, m = (v dt)^2).
//
// The GPU keeps mu = nu / (1 + e) instead of nu: then mu^k = (mu^{k+1} +
// w^{k+1}) / (1 + e) and psi = sum_a k_a [G_a mu^{k+1}](x + e_a) - [G_a
// mu^{k+1}](x - e_a) with G_a(y) = d_a(y+1)^2 - d_a(y-1)^2, both computed by the
// adjoint step kernel at its PML tiles (mu is zero off the PML).  The time sum
// sum_k w^k g^{k-1} runs in fp32 per point over blocks of FOLD_EVERY steps
// (counted from step 0, so the grouping does not depend on the checkpoint
// interval) and is folded into an fp64 sum after each block.
#pragma once

namespace {

// The adjoint step's configuration for tile shape C: five tiles per plane, two stages.
template <class C>
using AdjCfg = TileCfg<C::TXT, C::TYT, C::TY, C::NU, 2, C::MINB>;
constexpr int FOLD_EVERY = 32;

// G += S, S = 0 over the padded arrays (the fp64 time sum of the gradient).
__global__ void fold_kernel(float *__restrict__ S, double *__restrict__ G, long long n)
{
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        G[q] += (double)S[q];
        S[q] = 0.0f;
    }
}

// J = 1/2 sum (traces - observed)^2 in fp64, in a fixed order (two passes:
// per-block partial sums, then one block of as many threads), so repeated runs
// agree to the bit.
constexpr int MISFIT_BLOCKS = 256;

__global__ void misfit_partial_kernel(const float *__restrict__ tr, const float *__restrict__ obs,
                                      long long n, double *partial)
{
    __shared__ double ws[8];
    double s = 0.0;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        const double d = (double)tr[q] - (double)obs[q];
        s += 0.5 * d * d;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
        partial[blockIdx.x] = t;
    }
}

__global__ void misfit_final_kernel(const double *partial, double *J)
{
    __shared__ double ws[MISFIT_BLOCKS / 32];
    double t = partial[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        t = 0.0;
        for (int w = 0; w < MISFIT_BLOCKS / 32; ++w) t += ws[w];
        *J = t;
    }
}

// dJ/dv = 2 (sum_k w^k g^{k-1}) / v on the compact grid, planes in grid.y.  fp64
// division is slow here (87 us at 128^3): 1 / v comes from the fp32 reciprocal
// and one Newton step in fp64 (relative error below 2^-46), the quotient from a
// product and its residual (Markstein, IBM J. Res. Dev. 34, 1990), which leaves an
// error of half a unit in the last place, as the division did; the indices come
// from one 32-bit division.
__global__ void chain_kernel(PadGeom g, const double *__restrict__ G,
                             const float *__restrict__ vel, double *__restrict__ grad_v, int j0,
                             int rows)
{
    const uint32_t items = uint32_t(g.Nx) * uint32_t(rows);
    for (int k = blockIdx.y; k < g.Nz; k += gridDim.y) {
        const long long c0 = ((long long)k * g.Ny + j0) * g.Nx, p0 = g.origin + k * g.sxy + j0 * g.sx;
        for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < items; t += gridDim.x * blockDim.x) {
            const uint32_t j = t / uint32_t(g.Nx), i = t - j * uint32_t(g.Nx);
            const float v = vel[c0 + t];
            double inv = (double)__frcp_rn(v);
            inv = fma(inv, fma(-(double)v, inv, 1.0), inv);
            if (!(v > 1e-30f && v < 1e30f)) inv = 1.0 / (double)v;  // no fp32 reciprocal there
            const double num = 2.0 * G[p0 + j * g.sx + i], quo = num * inv;
            // an infinite quotient has no residual
            grad_v[c0 + t] = isfinite(quo) ? fma(fma(-(double)v, quo, num), inv, quo) : quo;
        }
    }
}

int adjoint_prepared = 0;
int adjoint_occ = 0;  // resident adjoint-step CTAs per SM

}  // namespace

extern "C" int adjoint_shot(const sgb_grid *g, const float *velocity, const float *wavelet,
                            int32_t nt, const int32_t *src_ijk, const int32_t *rec_ijk,
                            int32_t nrec, const float *observed, int32_t ckpt_every,
                            double *misfit_out, double *grad_velocity, void *stream)
{
    sgb_layout_info L;
    int rc = check_grid(g, &L);
    if (rc) return rc;
    if (g->storage != SGB_FP32) return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: SGB_FP32 only");
    if (!velocity || !wavelet || !src_ijk || !rec_ijk || !observed || !misfit_out || !grad_velocity)
        return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: NULL argument");
    if (nt < 1 || nrec < 1) return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: nt and nrec must be >= 1");
    if (ckpt_every < 0) return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: ckpt_every < 0");
    const int C = ckpt_every == 0 ? 100 : std::min<int>(ckpt_every, nt);
    if (!in_inner(g, src_ijk[0], src_ijk[1], src_ijk[2]))
        return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: source outside the inner region");
    std::vector<long long> off(nrec);
    for (int r = 0; r < nrec; ++r) {
        const int i = rec_ijk[3 * r], j = rec_ijk[3 * r + 1], k = rec_ijk[3 * r + 2];
        if (!in_inner(g, i, j, k))
            return fail(SGB_ERR_INVALID_ARG, "adjoint_shot: receiver %d outside the inner region", r);
        off[r] = L.origin + (long long)k * L.stride_z + (long long)j * L.sx + i;
    }
    DevState *ds;
    if ((rc = device_state(&ds))) return rc;
    if (!adjoint_prepared) {
        std::lock_guard<std::mutex> lk(g_mu);
        int occ_acc = 0, occ_adj = 0;
        for (const bool square : {false, true}) {
            rc = with_tile(StepGrid{0, square}, [&](auto c) {
                using C = decltype(c);
                using A = AdjCfg<C>;
                const int e = prepare_kernel<C>(fwd_acc_kernel<C>, Stage<C, float, MODE_FWD_ACC>::SMEM_BYTES,
                                                &occ_acc);
                return e ? e : prepare_kernel<A>(adjoint_step_kernel<A>, Stage<A, float, MODE_ADJ>::SMEM_BYTES,
                                                 &occ_adj);
            });
            if (rc) return rc;
        }
        adjoint_occ = occ_adj;
        adjoint_prepared = 1;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const long long ncomp = (long long)L.Nx * L.Ny * L.Nz;
    const size_t fbytes = (size_t)L.elems * 4;
    const int nseg = (nt + C - 1) / C;
    Scratch sc{st, ds->pool, {}};
    // inputs on the device
    auto to_dev = [&](const void *src, size_t bytes, void **dst) -> int {
        if (is_device_ptr(src)) {
            *dst = const_cast<void *>(src);
            return SGB_OK;
        }
        int r2 = sc.get(dst, bytes);
        if (r2) return r2;
        CUDA_TRY(cudaMemcpyAsync(*dst, src, bytes, cudaMemcpyHostToDevice, st));
        return SGB_OK;
    };
    float *d_vel, *d_wav, *d_obs;
    if ((rc = to_dev(velocity, (size_t)ncomp * 4, (void **)&d_vel)) ||
        (rc = to_dev(wavelet, (size_t)nt * 4, (void **)&d_wav)) ||
        (rc = to_dev(observed, (size_t)nt * nrec * 4, (void **)&d_obs)))
        return rc;
    // m, and the CFL check against the model's maximum
    float *m;
    int *d_range, *d_err;  // d_err: this call's device error word, so concurrent calls stay independent
    if ((rc = get_call_words(sc, st, &d_range, &d_err)) || (rc = sc.get((void **)&m, fbytes)) ||
        (rc = make_model(g, L, st, d_vel, m, d_range)))
        return rc;
    // fields
    // fields that start at zero, in one block: the fp64 sum, then u0, u1, phi (the
    // state that a checkpoint holds) and the adjoint's w0, w1, mu0, mu1, S
    float *fields, *ck, *seg, *d_tr;
    double *gsum64, *d_J;
    long long *d_off;
    const int nck = std::max(0, nseg - 2);  // checkpoints of segments 1 .. nseg - 2 (see below)
    if ((rc = sc.get((void **)&gsum64, (size_t)L.elems * 8 + 8 * fbytes)) ||
        (rc = sc.get((void **)&ck, fbytes * 3 * (size_t)nck)) ||
        (rc = sc.get((void **)&seg, fbytes * (size_t)C)) ||
        (rc = sc.get((void **)&d_tr, (size_t)nt * nrec * 4)) || (rc = sc.get((void **)&d_J, 8)) ||
        (rc = sc.get((void **)&d_off, (size_t)nrec * 8)))
        return rc;
    fields = reinterpret_cast<float *>(gsum64 + L.elems);
    float *f[8];
    for (int q = 0; q < 8; ++q) f[q] = fields + (size_t)q * L.elems;
    float *u0 = f[0], *u1 = f[1], *phi = f[2], *w0 = f[3], *w1 = f[4], *mu0 = f[5], *mu1 = f[6],
          *gsum = f[7];
    CUDA_TRY(cudaMemcpyAsync(d_off, off.data(), (size_t)nrec * 8, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemsetAsync(gsum64, 0, (size_t)L.elems * 8 + 8 * fbytes, st));

    StepArgs base;
    fill_step_constants(g, L, base);
    base.phi = phi;
    base.err = d_err;
    base.si = src_ijk[0];
    base.sj = src_ijk[1];
    base.sk = src_ijk[2];
    base.wavelet = d_wav;
    const StepGrid sg = choose_decomposition<float>(ds->sms, ds->occ, base);
    float *ubuf[2] = {u0, u1};  // ubuf[0] = u^{-1}, ubuf[1] = u^0
    StepMaps fmaps[2];
    for (int p = 0; p < 2; ++p)
        if ((rc = encode_step_maps<float>(fmaps[p], ubuf[(p + 1) & 1], ubuf[p & 1], m, phi, L, sg))) return rc;

    // 1. forward with checkpoints (u^n, u^{n-1}, phi^n before step n = s C).  The
    // last segment stores its g^n as it goes, so the backward sweep starts there
    // without recomputing it, and the first one starts from zero: neither needs a
    // checkpoint (two segments of 50 steps at 128^3: 4.26 -> 3.60 ms).
    const size_t state_bytes = 3 * fbytes;
    const int n_last = (nseg - 1) * C;
    auto checkpoint = [&](int sg) { return ck + (size_t)(sg - 1) * 3 * L.elems; };
    auto step_acc = [&](int n, int na, bool sample) -> int {  // step n, keeping g^n
        StepArgs a = base;
        a.u_out = ubuf[n & 1];
        a.u_cur = ubuf[(n + 1) & 1];
        a.step_add = n;
        a.acc_out = seg + (size_t)(n - na) * L.elems;
        if (sample) {
            a.nrec = nrec;
            a.rec_off = d_off;
            a.traces = d_tr;
        }
        const StepMaps &mp = fmaps[n & 1];
        CUDA_TRY(with_tile(sg, [&](auto c) {
            using C = decltype(c);
            return launch_dependent(fwd_acc_kernel<C>, sg.ctas, C::BLOCK,
                                    Stage<C, float, MODE_FWD_ACC>::SMEM_BYTES, st, a, mp.ucur,
                                    mp.ucur_in, mp.uprev, mp.m, mp.phi);
        }));
        ++t_launches;
        return SGB_OK;
    };
    for (int n = 0; n < nt; ++n) {
        if (n >= n_last) {
            if ((rc = step_acc(n, n_last, true))) return rc;
            continue;
        }
        if (n > 0 && n % C == 0)
            CUDA_TRY(cudaMemcpyAsync(checkpoint(n / C), u0, state_bytes, cudaMemcpyDeviceToDevice, st));
        StepArgs a = base;
        a.u_out = ubuf[n & 1];
        a.u_cur = ubuf[(n + 1) & 1];
        a.step_add = n;
        a.nrec = nrec;
        a.rec_off = d_off;
        a.traces = d_tr;
        if ((rc = launch_step<float>(a, fmaps[n & 1], sg, st))) return rc;
    }
    gather_kernel<<<(nrec + 255) / 256, 256, 0, st>>>(ubuf[(nt - 1) & 1], d_off, nrec,
                                                      d_tr + (size_t)(nt - 1) * nrec, d_err);
    CUDA_TRY(cudaGetLastError());
    double *d_part;
    if ((rc = sc.get((void **)&d_part, MISFIT_BLOCKS * 8))) return rc;
    misfit_partial_kernel<<<MISFIT_BLOCKS, 256, 0, st>>>(d_tr, d_obs, (long long)nt * nrec, d_part);
    CUDA_TRY(cudaGetLastError());
    misfit_final_kernel<<<1, MISFIT_BLOCKS, 0, st>>>(d_part, d_J);
    CUDA_TRY(cudaGetLastError());

    // 2. backward sweep, segment by segment from the last
    float *wbuf[2] = {w0, w1};  // w^k lives in wbuf[k & 1]
    float *mbuf[2] = {mu0, mu1};  // mu^k lives in mbuf[k & 1]
    StepArgs abase = base;
    abase.sk = -1;  // the adjoint's sources are the receivers
    abase.gsum = gsum;
    const StepGrid ag = choose_decomposition<float>(ds->sms, adjoint_occ, abase);
    const int box_x = ag.square ? CfgSq::BX : Cfg::BX, box_y = ag.square ? CfgSq::BY : Cfg::BY;
    std::vector<CUtensorMap> acc_maps(C);
    for (int q = 0; q < C; ++q)
        if ((rc = encode_map<float>(&acc_maps[q], seg + (size_t)q * L.elems, L, box_x, box_y))) return rc;
    // [k & 1]: reads w^{k+1} = wbuf[(k+1)&1] and mu^{k+1}, writes wbuf[k&1]
    StepMaps amaps[2];
    for (int p = 0; p < 2; ++p) {
        if ((rc = encode_step_maps<float>(amaps[p], wbuf[(p + 1) & 1], wbuf[p & 1], m,
                                          mbuf[(p + 1) & 1], L, ag)))
            return rc;
        // mu^{k+1} as a box with its x-y neighbours (x halo 4, y halo 1)
        rc = with_tile(ag, [&](auto c) {
            using GA = Stage<AdjCfg<decltype(c)>, float, MODE_ADJ>;
            return encode_map<float>(&amaps[p].phi, mbuf[(p + 1) & 1], L, GA::MBW, GA::MBH, SGB_L2PROMO);
        });
        if (rc) return rc;
    }
    CUtensorMap gs_map;
    if ((rc = encode_map<float>(&gs_map, gsum, L, box_x, box_y))) return rc;
    // receivers grouped by the unit that computes them, and in a unit by point (the
    // residuals of receivers at one point are added by one thread)
    UnitReceivers ur;
    int *d_rs, *d_ri;
    long long *d_ro;
    with_tile(ag, [&](auto c) { group_receivers<decltype(c)>(abase, ag.ctas, rec_ijk, nrec, ur); });
    const auto by_point = [&](int p, int q) { return off[p] < off[q]; };
    for (int u = 0; u < ag.ctas; ++u) {
        const auto r0 = ur.list.begin() + ur.start[u], r1 = ur.list.begin() + ur.start[u + 1];
        if (!std::is_sorted(r0, r1, by_point)) std::stable_sort(r0, r1, by_point);
    }
    std::vector<long long> uoff(nrec);
    for (int q = 0; q < nrec; ++q) uoff[q] = off[ur.list[q]];
    if ((rc = sc.get((void **)&d_rs, ur.start.size() * 4)) || (rc = sc.get((void **)&d_ri, (size_t)nrec * 4)) ||
        (rc = sc.get((void **)&d_ro, (size_t)nrec * 8)))
        return rc;
    CUDA_TRY(cudaMemcpyAsync(d_rs, ur.start.data(), ur.start.size() * 4, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemcpyAsync(d_ri, ur.list.data(), (size_t)nrec * 4, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemcpyAsync(d_ro, uoff.data(), (size_t)nrec * 8, cudaMemcpyHostToDevice, st));
    abase.rec_start = d_rs;
    abase.rec_idx = d_ri;
    abase.rec_off = d_ro;
    abase.m_all = m;
    for (int q = 0; q < 3; ++q) {
        abase.rec_lo[q] = abase.rec_hi[q] = rec_ijk[q];
        for (int r = 1; r < nrec; ++r) {
            abase.rec_lo[q] = std::min(abase.rec_lo[q], rec_ijk[3 * r + q]);
            abase.rec_hi[q] = std::max(abase.rec_hi[q], rec_ijk[3 * r + q]);
        }
    }
    const int fgrid = ew_grid(L.elems, *ds);
    for (int s = nseg - 1; s >= 0; --s) {
        const int na = s * C, nbnd = std::min(na + C, nt);
        if (s == 0 && nseg > 1) CUDA_TRY(cudaMemsetAsync(u0, 0, state_bytes, st));
        else if (s < nseg - 1)
            CUDA_TRY(cudaMemcpyAsync(u0, checkpoint(s), state_bytes, cudaMemcpyDeviceToDevice, st));
        if (s < nseg - 1)
            for (int n = na; n < nbnd; ++n)  // recompute
                if ((rc = step_acc(n, na, false))) return rc;
        for (int k = nbnd; k >= na + 1; --k) {  // adjoint steps
            StepArgs a = abase;
            a.u_out = wbuf[k & 1];
            a.u_cur = wbuf[(k + 1) & 1];
            a.phi = mbuf[k & 1];
            a.mu_in = mbuf[(k + 1) & 1];
            a.acc_in = seg + (size_t)(k - 1 - na) * L.elems;
            a.tr_row = d_tr + (size_t)(k - 1) * nrec;
            a.obs_row = d_obs + (size_t)(k - 1) * nrec;
            a.step_add = k;
            const StepMaps &mp = amaps[k & 1];
            CUDA_TRY(with_tile(ag, [&](auto c) {
                using A = AdjCfg<decltype(c)>;
                return launch_dependent(adjoint_step_kernel<A>, ag.ctas, A::BLOCK,
                                        Stage<A, float, MODE_ADJ>::SMEM_BYTES, st, a, mp.ucur,
                                        mp.ucur_in, mp.uprev, mp.m, mp.phi, acc_maps[k - 1 - na],
                                        gs_map);
            }));
            ++t_launches;
            if ((k - 1) % FOLD_EVERY == 0) {  // blocks of steps counted from step 0
                fold_kernel<<<fgrid, 256, 0, st>>>(gsum, gsum64, (long long)L.elems);
                CUDA_TRY(cudaGetLastError());
                ++t_launches;
            }
        }
    }
    // 3. chain rule to velocity, outputs
    double *d_gv = grad_velocity;
    const bool host_gv = !is_device_ptr(grad_velocity);
    if (host_gv && (rc = sc.get((void **)&d_gv, (size_t)ncomp * 8))) return rc;
    CUDA_TRY(for_row_slabs(L.Ny, L.Nx, [&](int j0, int rows) {
        chain_kernel<<<conv_grid((long long)L.Nx * rows, L.Nz), CONV_THREADS, 0, st>>>(
            pad_geom(L), gsum64, d_vel, d_gv, j0, rows);
    }));
    if (host_gv)
        CUDA_TRY(cudaMemcpyAsync(grad_velocity, d_gv, (size_t)ncomp * 8, cudaMemcpyDeviceToHost, st));
    double J = 0.0;
    CUDA_TRY(cudaMemcpyAsync(&J, d_J, 8, cudaMemcpyDeviceToHost, st));
    int dev_err = 0;
    CUDA_TRY(cudaMemcpyAsync(&dev_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    *misfit_out = J;
    if (dev_err & DEV_ERR_TIMEOUT) return fail(SGB_ERR_TIMEOUT, "a kernel wait timed out");
    return SGB_OK;
}
