// A field record that names a neighbour outside the grid (a damaged record:
// the library builds none) ends the particle with the request's error flag
// before anything is read there.  Linked against libmp.so; the record of the
// last of four cells in a row is changed to name an active neighbour across
// its outer face, then put back.
#include <cstdio>
#include <vector>

#include "mp.h"
#include "mp_internal.h"

#define OK(call)                                                             \
    do {                                                                     \
        const int rc_ = (call);                                              \
        if (rc_ != 0) {                                                      \
            printf("%s: %d %s\n", #call, rc_, mp_last_error());              \
            return 2;                                                        \
        }                                                                    \
    } while (0)

int main()
{
    const double d4[4] = {1, 1, 1, 1}, qx[5] = {1, 1, 1, 1, 1}, q0[8] = {0};
    const double por[4] = {0.5, 0.5, 0.5, 0.5};
    const int8_t ib[4] = {1, 1, 1, 1};
    mp_ctx* ctx = nullptr;
    OK(mp_ctx_create(0, &ctx));
    mp_field_desc fd{1, 1, 4, d4, d4, d4, {0, 0, 0}, qx, q0, q0, por, ib, 0};
    mp_field* f = nullptr;
    OK(mp_field_load(ctx, &fd, &f));
    const mp::DevField& v = *mp::field_device_view(f);
    mp::CellF64 r64;
    mp::CellF32 r32;
    OK(cudaMemcpy(&r64, v.rec64 + 3, sizeof r64, cudaMemcpyDeviceToHost));
    OK(cudaMemcpy(&r32, v.rec32 + 3, sizeof r32, cudaMemcpyDeviceToHost));
    const int n = 23;
    std::vector<int32_t> cell(n);
    std::vector<double> local(3 * n, 0.5);
    for (int i = 0; i < n; ++i) cell[i] = i % 4;
    int bad = 0;
    for (int damaged = 1; damaged >= 0; --damaged) {
        mp::CellF64 a = r64;
        mp::CellF32 b = r32;
        if (damaged) {
            a.nb = (a.nb & ~(3ULL << 2)) | ((unsigned long long)mp::NB_ACTIVE << 2);   // face x+
            b.nb = (b.nb & ~(3u << 2)) | ((unsigned)mp::NB_ACTIVE << 2);
        }
        OK(cudaMemcpy(const_cast<mp::CellF64*>(v.rec64) + 3, &a, sizeof a, cudaMemcpyHostToDevice));
        OK(cudaMemcpy(const_cast<mp::CellF32*>(v.rec32) + 3, &b, sizeof b, cudaMemcpyHostToDevice));
        for (int prec : {MP_PREC_FP64, MP_PREC_MIXED}) {
            mp_release_desc rd{};
            rd.n = n;
            rd.kind = MP_RELEASE_EXPLICIT;
            rd.cell = cell.data();
            rd.local = local.data();
            mp_group* g = nullptr;
            OK(mp_release_group(ctx, f, &rd, nullptr, &g));
            mp_track_opts o{};
            o.mode = MP_MODE_ENDPOINT;
            o.precision = prec;
            o.schedule = MP_SCHED_DYNAMIC;
            o.t_stop = 1e30;
            mp_req r = 0;
            OK(mp_track(ctx, g, &o, nullptr, &r));
            mp_stats st{};
            OK(mp_get_stats(ctx, r, &st));
            const int want = damaged ? MP_ST_INVALID_RELEASE : MP_ST_EXIT_DOMAIN;
            mp_endpoints none{};
            const int rc = mp_get_endpoints(ctx, r, &none, 0, nullptr);
            if (st.device_error != damaged || st.n_status[want] != (uint64_t)n ||
                rc != (damaged ? MP_ERR_DEVICE : MP_OK)) {
                printf("precision %d damaged %d: error %d, %llu of %d with status %d, read %d\n", prec, damaged,
                       st.device_error, (unsigned long long)st.n_status[want], n, want, rc);
                bad = 1;
            }
            OK(mp_req_free(ctx, r));
            OK(mp_group_free(g));
        }
    }
    OK(mp_field_free(f));
    OK(mp_ctx_destroy(ctx));
    puts(bad ? "failed" : "ok");
    return bad;
}
