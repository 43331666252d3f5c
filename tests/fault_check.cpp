// GPU check of what a wait that runs out leaves behind (a block of a team that
// never arrives, polls limited to a moment; nothing faults or hangs), of a
// served job that ends with an error, and of a read without host memory.  The
// sources of the population and the server are part of this program, so that
// it reaches their arguments.
#include "population.cu"
#include "server.cu"

#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#define CHECK(x)                                                              \
    do {                                                                      \
        if (!(x)) {                                                           \
            std::printf("FAIL line %d: %s (%s)\n", __LINE__, #x, spg_last_error()); \
            std::exit(1);                                                     \
        }                                                                     \
    } while (0)

namespace {

constexpr uint32_t kLoci = 64, kCap = 32;

struct Inputs {
    std::vector<int16_t> effects = std::vector<int16_t>(kLoci);
    std::vector<uint32_t> table = std::vector<uint32_t>(kBins, 0xC0000000u);
    spg_pop_desc desc{};
    explicit Inputs(uint32_t n) {
        for (uint32_t l = 0; l < kLoci; ++l) effects[l] = (int16_t)((int)(l * 37u % 101u) - 50);
        desc.n = n;
        desc.n_loci = kLoci;
        desc.seed = n;
        desc.effects = effects.data();
        desc.p0_q32 = 0x80000000u;
        desc.surv_table = table.data();
        desc.bin_bias = 4096;
        desc.bin_shift = 2;
        desc.mu = 1e-3;
        desc.stats_capacity = kCap;
    }
};

// A launch of teams in which only `present` of the population's `team` blocks
// take part.
void launch_team(spg_pop *p, const std::vector<uint32_t> &present, uint32_t team) {
    static_assert(sizeof(SoloArgs) <= 1024, "the places follow the arguments");
    SoloArgs args = p->sa;
    args.barrier_tries = 1u << 12;
    std::vector<TeamPlace> places;
    std::vector<uint32_t> start(1, 0u);
    for (uint32_t r : present) {
        places.push_back(TeamPlace{0u, (uint16_t)r, (uint16_t)team});
        start.push_back((uint32_t)places.size());
    }
    char *mem = nullptr;
    CHECK(cudaMalloc(&mem, 4096) == cudaSuccess);
    CHECK(cudaMemcpy(mem, &args, sizeof args, cudaMemcpyHostToDevice) == cudaSuccess);
    CHECK(cudaMemcpy(mem + 1024, places.data(), places.size() * sizeof(TeamPlace), cudaMemcpyHostToDevice) == cudaSuccess);
    CHECK(cudaMemcpy(mem + 2048, start.data(), start.size() * 4, cudaMemcpyHostToDevice) == cudaSuccess);
    CHECK(cudaDeviceSynchronize() == cudaSuccess);
    TeamArgs t{};
    t.members = reinterpret_cast<const SoloArgs *>(mem);
    t.places = reinterpret_cast<const TeamPlace *>(mem + 1024);
    t.block_places = reinterpret_cast<const uint32_t *>(mem + 2048);
    t.n_gen = 1;
    t.keep_last = 1;
    SoloKernel k = team_kernel(team_kind(false, false, false));
    CHECK(prepare_solo(k) == SPG_OK);
    void *params[] = {&t};
    CHECK(cudaLaunchCooperativeKernel(k.fn, dim3((unsigned)present.size()), dim3(kSoloThreads), params, k.smem,
                                      p->stream) == cudaSuccess);
    CHECK(cudaStreamSynchronize(p->stream) == cudaSuccess);
    CHECK(cudaFree(mem) == cudaSuccess);
}

void set_status(const PopView &v, int32_t status) {
    CHECK(cudaStreamSynchronize(v.stream) == cudaSuccess);
    CHECK(cudaMemcpy(v.base + v.L.state + offsetof(DevState, status), &status, 4, cudaMemcpyHostToDevice) == cudaSuccess);
    CHECK(cudaDeviceSynchronize() == cudaSuccess);
}

struct Result {
    std::vector<spg_stats> stats = std::vector<spg_stats>(10);
    std::vector<uint32_t> counts = std::vector<uint32_t>(10 * kLoci), geno, surv;
    spg_state state{};
};
Result read(spg_pop *p) {
    Result r;
    uint32_t S = 0;
    r.geno.resize((size_t)p->n * 2 * p->words);
    r.surv.assign(p->n, 0u);
    CHECK(spg_read_stats(p, 4, 10, r.stats.data()) == SPG_OK);
    CHECK(spg_read_locus_counts(p, 4, 10, r.counts.data()) == SPG_OK);
    CHECK(spg_read_genotypes(p, r.geno.data(), r.geno.size()) == SPG_OK);
    CHECK(spg_read_survivors(p, r.surv.data(), r.surv.size(), &S) == SPG_OK);
    CHECK(spg_get_state(p, &r.state) == SPG_OK);
    return r;
}

spg_pop *create(const Inputs &in) {
    spg_pop *p = nullptr;
    CHECK(spg_create_population(&in.desc, nullptr, nullptr, &p) == SPG_OK);
    CHECK(spg_set_locus_counts(p, 1) == SPG_OK);
    CHECK(spg_step_generations(p, 3) == SPG_OK);
    return p;
}

// missing: the rank that does not arrive; it comes late, in a launch of its
// own.  counts: the restored run's per-locus counts are compared too.
void barrier(uint32_t n, uint32_t missing, bool counts) {
    const Inputs in(n);
    spg_pop *ref = create(in), *p = create(in);
    CHECK(spg_step_generations(ref, 10) == SPG_OK);
    const Result want = read(ref);
    size_t bytes = 0;
    CHECK(spg_checkpoint_size(p, &bytes) == SPG_OK);
    std::vector<char> saved(bytes);
    CHECK(spg_checkpoint(p, saved.data(), bytes) == SPG_OK);

    std::vector<uint32_t> present;
    for (uint32_t r = 0; r < 4; ++r)
        if (r != missing) present.push_back(r);
    spg_state st;
    launch_team(p, present, 4);
    CHECK(spg_get_state(p, &st) == SPG_OK && st.status == SPG_ERR_TIMEOUT && st.gen == 3);
    set_status(p->view(), SPG_OK);  // as a block saw it that started before the others gave up
    launch_team(p, {missing}, 4);
    CHECK(spg_get_state(p, &st) == SPG_OK && st.status == SPG_ERR_TIMEOUT && st.gen == 3);
    for (uint32_t k : {1u, 5u}) {  // later calls do nothing, and reads say why
        CHECK(spg_step_generations(p, k) == SPG_OK);
        CHECK(spg_get_state(p, &st) == SPG_OK && st.status == SPG_ERR_TIMEOUT && st.gen == 3);
    }
    std::vector<spg_stats> rec(3);
    CHECK(spg_read_stats(p, 1, 3, rec.data()) == SPG_ERR_TIMEOUT && rec[2].gen == 3);

    // a restored checkpoint runs as if nothing had happened
    CHECK(spg_restore(p, saved.data(), bytes) == SPG_OK);
    CHECK(spg_step_generations(p, 10) == SPG_OK);
    const Result got = read(p);
    CHECK(std::memcmp(got.stats.data(), want.stats.data(), want.stats.size() * sizeof(spg_stats)) == 0);
    CHECK(got.geno == want.geno && got.surv == want.surv);
    CHECK(got.state.gen == 13 && got.state.status == SPG_OK);
    CHECK(!counts || got.counts == want.counts);
    spg_destroy(p);
    spg_destroy(ref);
}

// A job whose device state says that a wait ran out is finished with that
// status; the others are not held up.
void served_job() {
    const Inputs a(5000), b(9000), c(700);
    spg_server_config cfg{};
    cfg.gens_per_tick = 4;
    spg_server *s = nullptr;
    CHECK(spg_server_create(&cfg, nullptr, nullptr, &s) == SPG_OK);
    uint64_t job[3];
    const Inputs *in[3] = {&a, &b, &c};
    for (int i = 0; i < 3; ++i) CHECK(spg_server_submit(s, &in[i]->desc, nullptr, 20, 0.0, job + i) == SPG_OK);
    CHECK(spg_server_tick(s, nullptr, nullptr) == SPG_OK);
    set_status(s->jobs[job[1]]->v, SPG_ERR_TIMEOUT);
    CHECK(spg_server_drain(s) == SPG_OK);
    std::vector<spg_stats> rec(20);
    for (int i = 0; i < 3; ++i) {
        spg_job_info info;
        CHECK(spg_server_job_info(s, job[i], &info) == SPG_OK && info.state == SPG_JOB_FINISHED);
        CHECK(info.status == (i == 1 ? SPG_ERR_TIMEOUT : SPG_OK) && info.gen == (i == 1 ? 4u : 20u));
        CHECK(spg_server_job_stats(s, job[i], 1, info.gen, rec.data()) == SPG_OK && rec[info.gen - 1].gen == info.gen);
    }
    spg_server_counters n;
    CHECK(spg_server_stats(s, &n) == SPG_OK && n.memory_used == 0 && n.resident == 0);
    spg_server_destroy(s);
}

// Reading statistics needs no host memory that may run out unreported.
bool g_no_memory = false;

void host_memory() {
    const Inputs in(1000);
    spg_pop *p = nullptr;
    CHECK(spg_create_population(&in.desc, nullptr, nullptr, &p) == SPG_OK);
    CHECK(spg_step_generations(p, 3) == SPG_OK);
    spg_stats rec[3];
    g_no_memory = true;
    const int rc = spg_read_stats(p, 1, 3, rec);
    g_no_memory = false;
    CHECK(rc == SPG_OK && rec[2].gen == 3);
    spg_destroy(p);
}

}  // namespace

void *operator new(size_t bytes) {
    void *p = g_no_memory ? nullptr : std::malloc(bytes);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "barrier")
        for (uint32_t missing : {0u, 2u}) barrier(20000, missing, false);
    else if (what == "counts") barrier(20000, 3, true);
    else if (what == "served") served_job();
    else if (what == "memory") host_memory();
    else return 2;
    std::printf("ok\n");
    return 0;
}
