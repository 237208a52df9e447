// The kernels as far as the fake runtime plays them: the state words, the final
// basis and the lane's rings, from the library's own structs.
#include <cuda_runtime.h>

#include <chrono>
#include <cstring>

#include "tsx_cluster.cuh"
#include "tsx_device.cuh"
#include "tsx_team.cuh"

extern "C" {
int fake_plan_status = 0, fake_plan_fail = 0, fake_plan_k = 0;
unsigned fake_team_next[2];   // k_team_solve: the list counters at its start
int fake_team_wide = 0;       // and its wide teams
int fake_team_size[512];      // blocks of each team (0: no such team)
int fake_lane_ms = 0;         // the lane's launch stays for this long, or until its stop word is set
}

namespace {
using tsx::DevState;
bool is(const char* name, const char* what) { return strstr(name, what) != nullptr; }
void set_basis(int* basis, int m, int n) {
    for (int i = 0; i < m; ++i) basis[i] = i < fake_plan_k ? i : n + i;
}
// Solves what the rings hold.
using Clock = std::chrono::steady_clock;
tsx::TeamServeParams<double> lane;
bool lane_open = false;
Clock::time_point lane_end;
void serve() {
    for (unsigned l = 0; l < 2; ++l)
        for (; lane.head[l] != __atomic_load_n(lane.ring.tail + l, __ATOMIC_ACQUIRE); ++lane.head[l]) {
            const unsigned slot = l * lane.cap + (lane.head[l] & (lane.cap - 1u));
            const tsx::TeamJob<double> J = lane.ring.jobs[slot];
            memset(J.st, 0, sizeof *J.st);
            set_basis(J.basis, J.m, J.n);
            J.st->status = fake_plan_status;
            __atomic_store_n(lane.ring.done + slot, lane.head[l] + 1u, __ATOMIC_RELEASE);
        }
}
void finish(DevState* st) {
    st->status = fake_plan_status;
    st->fail = fake_plan_fail;
    st->iters = 7;
}

}  // namespace

extern "C" void fake_play(const char* name, void** a) {
    if (is(name, "k_reset_state")) {
        DevState* st = *(DevState**)a[0];
        memset(st, 0, sizeof *st);
        st->status = tsx::kRunning;
    } else if (is(name, "k_build")) {
        set_basis(*(int**)a[8], *(int*)a[0], *(int*)a[1]);
    } else if (is(name, "k_pivot_delayed") || is(name, "k_pivot_overlap")) {
        finish(*(DevState**)a[3]);
    } else if (is(name, "k_pivot_persistent") || is(name, "k_ml_update")) {
        finish(((tsx::Params<double>*)a[0])->st);
    } else if (is(name, "k_cluster_solve")) {
        finish(((tsx::ClusterParams*)a[0])->st);
    } else if (is(name, "k_team_solve")) {
        auto* P = (tsx::TeamParams<double>*)a[0];
        memcpy(fake_team_next, P->next, sizeof fake_team_next);
        memset(fake_team_size, 0, sizeof fake_team_size);
        for (int t = 0; t < 512 && P->first + t < P->size; ++t) fake_team_size[t] = P->size[t];
        for (fake_team_wide = 0; P->first + fake_team_wide < P->size && P->list[fake_team_wide] == 1;) ++fake_team_wide;
        for (int l = 0; l < 2; ++l)
            for (int k = 0; k < P->count[l]; ++k) {
                const tsx::TeamJob<double>& J = P->jobs[P->order[l][k]];
                set_basis(J.basis, J.m, J.n);
                J.st->status = fake_plan_status;
            }
    } else if (is(name, "k_team_serve")) {
        lane = *(tsx::TeamServeParams<double>*)a[0];
        lane_end = Clock::now() + std::chrono::milliseconds(fake_lane_ms);
        lane_open = true;
        serve();
    }
}

// Whether a lane's launch is on the device (called with the runtime's lock).
extern "C" int fake_lane_running() {
    if (!lane_open) return 0;
    serve();
    lane_open = Clock::now() < lane_end && __atomic_load_n(lane.ring.stop, __ATOMIC_ACQUIRE) == 0;
    return lane_open;
}
