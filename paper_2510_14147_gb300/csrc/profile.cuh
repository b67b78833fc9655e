// profile.cuh -- stage timing scopes (see profile.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ct {

bool prof_on();
// Adds the stages recorded by this thread to the table (waits for their events).
void prof_flush();

class ProfScope {
  public:
    // calls: what the stage counts as (a forest: one build per tree)
    ProfScope(const char *name, cudaStream_t s, int64_t calls = 1);
    ~ProfScope();
    ProfScope(const ProfScope &) = delete;
    ProfScope &operator=(const ProfScope &) = delete;

  private:
    cudaStream_t s_;
    bool active_;
    int idx_ = -1;
};

}  // namespace ct
