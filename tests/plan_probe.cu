// Host-side planning of the sweep launches for contexts that exist nowhere: the plan
// depends on sizes only, so it can be checked over every size without a GPU.
#include <cstring>

#include "../paper_1212_3975_gb300/csrc/muca_internal.cuh"

namespace {
muca_ctx context(int model, int L, int p, int staging, int chains_per_block)
{
    muca_ctx c;
    std::memset(static_cast<void *>(&c), 0, sizeof(c));
    c.model = model;
    c.L = L;
    c.q = model == MUCA_ISING ? 2 : 8;
    c.p = p;
    c.p_pad = (p + 31) / 32 * 32;
    c.V = L * L;
    c.n_bins = muca::n_bins_of(model, L);
    c.n_de = muca::n_de_of(model);
    c.cfg.staging = staging;
    c.cfg.chains_per_block = chains_per_block;
    c.n_sm = 152;
    c.smem_per_sm = 228 * 1024;
    c.smem_reserved = 1024;
    c.row_words = model == MUCA_ISING ? (L + 31) / 32 : (L + 3) / 4;
    c.lat_words = L * c.row_words;
    return c;
}
}  // namespace

extern "C" {

// chains of a batch's work unit, sweeps of one of its launches at most
void probe_batch(int model, int L, int p, int out[2])
{
    const muca_ctx c = context(model, L, p, MUCA_STAGING_AUTO, 0);
    const muca::SweepPlan pl = muca::plan_sweeps(&c, false, muca::kBatchGroups);
    out[0] = muca::sweep_shape(&c, pl, true, muca::kBatchGroups).chains;
    out[1] = muca::batch_max_sweeps(&c);
}

// whether a standalone launch takes its staging; its shared memory and chains per block
int probe_launch(int model, int L, int p, int staging, int chains_per_block, int hist, int out[2])
{
    const muca_ctx c = context(model, L, p, staging, chains_per_block);
    const muca::SweepPlan pl = muca::plan_sweeps(&c);
    const muca::SweepShape s = muca::sweep_shape(&c, pl, hist != 0);
    out[0] = (int)s.smem;
    out[1] = s.chains;
    return muca::staging_fits(pl, s);
}

// status of a context whose sweeps set `fault`
int probe_fault(int fault)
{
    muca_ctx c = context(MUCA_ISING, 8, 1, MUCA_STAGING_AUTO, 0);
    c.h_fault = &fault;
    return muca::check_fault(&c);
}

int probe_launches(int n_sweeps, int split, int most) { return muca::sweep_launches(n_sweeps, split, most); }
}
