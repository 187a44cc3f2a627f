"""rosaq_last_status against a fake CUDA runtime on host memory (no GPU): whatever call fails while it cleans up behind a launch that
gave up, the status word stays set as long as anything of that launch is left, because a set word is what makes the next launch empty
its own slots."""
import shutil
import subprocess

import pytest

from paper_2506_13472_b200 import build as b

RUNTIME = r"""
#include <string.h>
int calls, fail_at;
static int step() { return ++calls == fail_at ? 999 : 0; }
extern "C" {
int cudaGetDevice(int *d) { return *d = 0, 0; }
int cudaSetDevice(int) { return 0; }
int cudaGetLastError() { return 0; }
int cudaStreamSynchronize(void *) { return step(); }
int cudaMemcpy(void *d, const void *s, size_t n, int) { return memcpy(d, s, n), step(); }
int cudaMemset(void *d, int v, size_t n) {
  const int e = step();
  if (!e) memset(d, v, n);
  return e;
}
void **__cudaRegisterFatBinary(void *) { return 0; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
}
"""
LOADER = r"""
#include <dlfcn.h>
#include <stdio.h>
int main(int, char **argv) {           // (lazily: what the test does not call stays undefined)
  void *lib = dlopen(argv[1], RTLD_LAZY);
  if (!lib) return fprintf(stderr, "%s\n", dlerror()), 2;
  return reinterpret_cast<int (*)()>(dlsym(lib, "run"))();
}
"""
MAIN = r"""
#include "rosaq_api.cu"
#include <stdio.h>
extern int calls, fail_at;
extern "C" int run() {
  for (fail_at = 0;; ++fail_at) {
    rosaq_ctx ctx{};
    ctx.sm_count = 4;
    std::vector<unsigned> exchange(64, 1), old(32, 1), ws(32, 1), sk(rosaq::kSkCounterInts, 1), sync(rosaq::kPlSyncWords, 1),
        flags(rosaq::kPfFlagsPerSm * 4, 1);
    int status[2] = {ROSAQ_ERR_TIMEOUT, 0};
    ctx.d_status = status;
    ctx.pl_exchange = reinterpret_cast<float *>(exchange.data()), ctx.pl_exchange_bytes = 256;
    ctx.retired[0] = old.data(), ctx.retired_exchange[0] = 128;
    ctx.retired[1] = ws.data(), ctx.retired_exchange[1] = 0;
    ctx.n_retired = 2;
    ctx.sk_arrive = reinterpret_cast<int *>(sk.data()), ctx.pl_sync = sync.data(), ctx.pf_flags = flags.data();
    calls = 0;
    const int st = rosaq_last_status(&ctx, nullptr);
    unsigned left = 0;
    for (unsigned v : exchange) left |= v ^ rosaq::kEmpty;
    for (unsigned v : old) left |= v ^ rosaq::kEmpty;
    for (const auto *x : {&sk, &sync, &flags})
      for (unsigned v : *x) left |= v;
    for (unsigned v : ws) left |= v ^ 1u;
    printf("%d %d %d %d %d\n", fail_at, calls, st, status[0], left != 0);
    if (fail_at > calls) return 0;
  }
}
"""


@pytest.mark.skipif(not shutil.which("nvcc"), reason="no nvcc")
def test_status_word_is_cleared_last(tmp_path):
    for name, text in (("main.cu", MAIN), ("runtime.cpp", RUNTIME), ("loader.cpp", LOADER)):
        (tmp_path / name).write_text(text)
    lib, exe = tmp_path / "lib.so", tmp_path / "loader"
    subprocess.run(["nvcc"] + b.NVCC_FLAGS + ["-shared", "-cudart", "none", "-o", lib, tmp_path / "main.cu", tmp_path / "runtime.cpp",
                                              "-Xlinker", "-z", "-Xlinker", "lazy"], check=True)
    subprocess.run(["g++", "-o", exe, tmp_path / "loader.cpp", "-ldl"], check=True)
    rows = [tuple(map(int, line.split())) for line in subprocess.run([exe, lib], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) > 6
    timeout = -6
    for fail_at, calls, st, word, left in rows:
        if fail_at == 0 or fail_at > calls:                          # nothing failed
            assert (st, word, left) == (timeout, 0, 0)
        else:
            assert st not in (0, timeout)
            assert word == timeout or not left, f"call {fail_at}: stale workspaces under a clear status"
