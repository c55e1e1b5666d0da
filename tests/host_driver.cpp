// The host driver of libmpr on the stand-in runtime (fake_cudart.cpp); test_host_driver.py builds it,
// names a scenario and reads what is printed: the status of the call, then the launches in order.
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <condition_variable>
#include <mutex>
#include <thread>

#include "fake_cudart.h"
#include "mpr.h"

namespace {

mpr_handle handle(int Lx, int Ly)
{
    std::vector<double> z((size_t)Lx * Ly, 0.5);
    std::vector<unsigned char> m((size_t)Lx * Ly, 1);
    mpr_handle h = nullptr;
    if (mpr_create(Lx, Ly, z.data(), m.data(), &h) != MPR_OK || mpr_set_temperature(h, 0.1) != MPR_OK) {
        fprintf(stderr, "%s\n", mpr_last_error());
        exit(1);
    }
    return h;
}

bool is_resident(const fake::Launch& l)
{
    return l.name.find("fine_kernel") != std::string::npos || l.name.find("coarse_kernel") != std::string::npos;
}

void report(mpr_status s)
{
    printf("status %d\n", (int)s);
    for (const fake::Launch& l : fake::launches)
        printf("%s programmatic=%d cooperative=%d grid=%u smem=%zu\n", l.name.c_str(), l.programmatic, l.cooperative,
               l.grid, l.smem);
}

}  // namespace

int main(int argc, char** argv)
{
    const char* const what = argc > 1 ? argv[1] : "";
    auto num = [&](int i) { return i < argc ? atoi(argv[i]) : 0; };
    if (!strcmp(what, "run")) {   // Lx Ly equil samples [sweep kernel]
        mpr_handle h = handle(num(2), num(3));
        if (argc > 6) mpr_set_sweep_kernel(h, num(6));
        fake::launches.clear();
        report(mpr_run(h, num(4), num(5)));
        mpr_destroy(h);
    } else if (!strcmp(what, "scarce")) {   // Lx Ly equil samples func: no allocation above 300 bytes
        mpr_handle h = handle(num(2), num(3));
        mpr_options o;
        mpr_get_options(h, &o);
        o.func = num(6);
        if (mpr_set_options(h, &o) != MPR_OK || mpr_set_temperature(h, 0.1) != MPR_OK) return 1;
        mpr_info before, after;
        mpr_get_info(h, &before);
        fake::launches.clear();
        fake::alloc_limit = 300;
        const mpr_status s = mpr_run(h, num(4), num(5));
        mpr_get_info(h, &after);
        report(s);
        if (!fake::refused_allocs || after.device_bytes > before.device_bytes + 300) return 1;
        mpr_destroy(h);
    } else if (!strcmp(what, "tune")) {   // Lx Ly n_eq n_meas
        mpr_handle h = handle(num(2), num(3));
        mpr_tuning t{num(4), num(5), 0.1, 1.0, 0.0, 1.5, 4};
        mpr_set_tuning(h, &t);
        fake::launches.clear();
        double T;
        report(mpr_tune_temperature(h, &T));
        mpr_destroy(h);
    } else if (!strcmp(what, "other")) {   // Lx Ly, and Lx Ly of a handle that runs before each resident launch
        mpr_handle h = handle(num(2), num(3)), g = handle(num(4), num(5));
        fake::launches.clear();
        bool inside = false;
        fake::on_launch = [&](const fake::Launch& l) {
            if (inside || !is_resident(l)) return 0;
            inside = true;
            mpr_status s = MPR_OK;
            std::thread([&] { s = mpr_run(g, 50, 0); }).join();
            inside = false;
            return s == MPR_OK ? 0 : (int)cudaErrorUnknown;
        };
        report(mpr_run(h, 50, 40));
        fake::on_launch = nullptr;
        mpr_destroy(h);
        mpr_destroy(g);
    } else if (!strcmp(what, "busy")) {   // Lx Ly, number of other handles that are in a run meanwhile
        mpr_handle h = handle(num(2), num(3));
        std::vector<mpr_handle> others;
        for (int i = 0; i < num(4); ++i) others.push_back(handle(40, 40));
        std::vector<std::thread> ts;
        std::mutex mu;
        std::condition_variable cv;
        int waiting = 0;
        bool go = false;
        const std::thread::id me = std::this_thread::get_id();
        fake::on_launch = [&](const fake::Launch&) {   // the others stop at their first launch
            if (std::this_thread::get_id() == me) return 0;
            std::unique_lock<std::mutex> lock(mu);
            ++waiting;
            cv.notify_all();
            cv.wait(lock, [&] { return go; });
            return 0;
        };
        for (mpr_handle g : others) ts.emplace_back([g] { mpr_run(g, 1, 0); });
        {
            std::unique_lock<std::mutex> lock(mu);
            cv.wait(lock, [&] { return waiting == (int)others.size(); });
        }
        fake::launches.clear();
        report(mpr_run(h, 5, 4));
        {
            std::lock_guard<std::mutex> lock(mu);
            go = true;
        }
        cv.notify_all();
        for (std::thread& t : ts) t.join();
        fake::on_launch = nullptr;
        fake::launches.clear();
        if (mpr_run(h, 5, 4) != MPR_OK) return 1;
        if (num(2) * num(3) <= 1400 * 1200 && !is_resident(fake::launches.front())) return 1;   // alone again
        for (mpr_handle g : others) mpr_destroy(g);
        mpr_destroy(h);
    } else if (!strcmp(what, "tags")) {   // Lx Ly of a lattice on a grid: sweeps until the tags start again
        // the first fields of resident::Args (mpr_resident.h)
        struct Args {
            int dims[8];
            void* arrays[10];
            float* er;
            unsigned long long* halo;
            uint32_t epoch;
            int nsweeps;
        };
        mpr_handle h = handle(num(2), num(3));
        uint64_t next = 0;   // tags up to here are taken
        int restarts = 0;
        bool ok = true;
        fake::on_launch = [&](const fake::Launch& l) {
            if (!is_resident(l)) return 0;
            const Args& a = *static_cast<const Args*>(l.args[0]);
            ok &= a.halo != nullptr && a.dims[0] == num(2) && a.dims[1] == num(3) && a.nsweeps >= 2;
            if (a.epoch < next) {   // tags start again: no word of an earlier launch is left
                ok &= a.epoch == 0 && *a.halo == 0;
                ++restarts;
            }
            *a.halo = ~0ull;   // what a launch leaves
            next = (uint64_t)a.epoch + 2ull * (uint64_t)a.nsweeps + 1;   // an exchange per pass, at most
            ok &= next < (1ull << 32);
            fake::launches.clear();
            return 0;
        };
        const mpr_status s = mpr_run(h, 1500000000, 0);
        fake::on_launch = nullptr;
        report(s);
        if (!ok || restarts != 1) {
            fprintf(stderr, "ok %d, restarts %d\n", ok, restarts);
            return 1;
        }
        mpr_destroy(h);
    } else if (!strcmp(what, "refuse")) {   // Lx Ly, error code of the resident launches
        mpr_handle h = handle(num(2), num(3));
        fake::launches.clear();
        fake::on_launch = [&](const fake::Launch& l) { return is_resident(l) ? num(4) : 0; };
        report(mpr_run(h, 5, 4));
        fake::on_launch = nullptr;
        mpr_destroy(h);
    } else {
        return 2;
    }
    return 0;
}
