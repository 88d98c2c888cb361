// The network's host code on the stand-in runtime: what its device buffers are after an allocation has failed.
#include "mlp.cu"

#include <cstdio>
#include <cstdlib>

extern long fake_fail_in, fake_null_copies;
size_t fake_live();

void mess_set_error(const char*, ...) {}
mess_status mess_basis_gpu(mess_basis*) { return MESS_EINVAL; }
mess_status mess_batch_basis(int, const mess_basis* const*, mess_basis**) { return MESS_EINVAL; }
void mess_free_basis(mess_basis*) {}
mess_status mess_scf_batch_density(mess_basis*, const mess_scf_opts*, mess_scf_result*, double*) { return MESS_EINVAL; }

static mess_status pass(mess_mlp* m, long long rows)
{
    std::vector<float> X(rows * DIN, 0.f), T(rows * DOUT, 0.f), M(rows * DOUT, 1.f), g(MlpParams::N);
    double loss = 0.0;
    return mess_mlp_loss_grad(m, rows, X.data(), T.data(), M.data(), &loss, g.data());
}

static bool whole(const mess_mlp* m, size_t rows)
{
    const size_t w = rows * WID;
    auto ok = [](const auto& d, size_t n) { return d.p && d.n >= n; };
    return ok(m->in, rows * (DIN + 2 * DOUT)) && ok(m->xb, rows * DIN) && ok(m->a1, w) && ok(m->a2, w) &&
           ok(m->dyb, rows * DOUT_PAD) && ok(m->dz2, w) && ok(m->dz1, w) && ok(m->z1, w) && ok(m->z2, w) &&
           ok(m->y, rows * DOUT_PAD) && ok(m->part, 1);
}

// For k = 0, 1, ... a new network takes a pass of 36 rows, one of 1000 in which allocation k fails, and one of 36;
// prints "k status-of-the-second status-of-the-third buffers-whole", until no allocation is left to fail.  Then the
// copies that met a null pointer, and the allocations still held once the networks are gone.
int main()
{
    for (long k = 0; k < 64; ++k) {
        mess_mlp* m = nullptr;
        if (mess_mlp_create(1, &m) != MESS_OK || pass(m, 36) != MESS_OK) return 2;
        fake_fail_in = k;
        const mess_status second = pass(m, 1000);
        const bool failed = fake_fail_in < 0;
        fake_fail_in = -1;
        const mess_status third = pass(m, 36);
        printf("%ld %d %d %d\n", k, (int)second, (int)third, (int)whole(m, 36));
        mess_mlp_destroy(m);
        if (!failed) break;
    }
    printf("null %ld\nheld %zu\n", fake_null_copies, fake_live());
    return 0;
}
