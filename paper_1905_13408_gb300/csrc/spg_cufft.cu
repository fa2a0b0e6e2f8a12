#include <dlfcn.h>

#include <mutex>

#include "spg_cufft.h"

namespace spg {

const CufftApi &cufft_api()
{
    static CufftApi c;
    static std::once_flag once;
    std::call_once(once, [] {
        const char *names[] = {"libcufft.so.12", "libcufft.so", "/usr/local/cuda/lib64/libcufft.so.12"};
        void *h = nullptr;
        for (const char *n : names)
            if ((h = dlopen(n, RTLD_NOW | RTLD_LOCAL))) break;
        if (!h) return;
        c.create = reinterpret_cast<decltype(c.create)>(dlsym(h, "cufftCreate"));
        c.set_auto_allocation =
            reinterpret_cast<decltype(c.set_auto_allocation)>(dlsym(h, "cufftSetAutoAllocation"));
        c.make_plan3d = reinterpret_cast<decltype(c.make_plan3d)>(dlsym(h, "cufftMakePlan3d"));
        c.set_work_area = reinterpret_cast<decltype(c.set_work_area)>(dlsym(h, "cufftSetWorkArea"));
        c.plan_many = reinterpret_cast<decltype(c.plan_many)>(dlsym(h, "cufftPlanMany"));
        c.set_stream = reinterpret_cast<decltype(c.set_stream)>(dlsym(h, "cufftSetStream"));
        c.exec_r2c = reinterpret_cast<decltype(c.exec_r2c)>(dlsym(h, "cufftExecR2C"));
        c.exec_c2r = reinterpret_cast<decltype(c.exec_c2r)>(dlsym(h, "cufftExecC2R"));
        c.exec_c2c = reinterpret_cast<decltype(c.exec_c2c)>(dlsym(h, "cufftExecC2C"));
        c.destroy = reinterpret_cast<decltype(c.destroy)>(dlsym(h, "cufftDestroy"));
        c.ok = c.create && c.set_auto_allocation && c.make_plan3d && c.set_work_area && c.plan_many && c.set_stream && c.exec_r2c && c.exec_c2r && c.exec_c2c && c.destroy;
    });
    return c;
}

}  // namespace spg
