"""How many CTA pairs the persistent launches count on: what the runtime answers
for the current device once the kernel's shared-memory limit has been raised
(it answers 0 before).  A C program stands in for the runtime, so that the
answers differ from half the SMs, and from device to device, without a GPU."""
import subprocess

import pytest

PROGRAM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
static int device, raised[2];
static const int answer[2] = {44, 30};
static int word;
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { *v = 100; return 0; }   /* SMs */
int cudaMalloc(void** p, size_t n) { *p = &word; return 0; }
int cudaMemset(void* p, int v, size_t n) { return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaGetLastError(void) { return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int v) {
    raised[device] = v;
    return 0;
}
int cudaOccupancyMaxActiveClusters(int* n, const void* f, const void* config) {
    *n = raised[device] > 48 * 1024 ? answer[device] : 0;
    return 0;
}

/* The schedule of T pair tiles on P clusters has 1 + P (T + P + 1) words. */
static int clusters(size_t words, size_t T) {
    for (size_t P = 1; P <= T; ++P)
        if (1 + P * (T + P + 1) == words) return (int)P;
    return -1;
}

int main(int argc, char** argv) {
    void* lib = dlopen(argv[1], RTLD_NOW);
    if (!lib) return fprintf(stderr, "%s\n", dlerror()), 2;
    size_t (*words)(int64_t, int64_t) =
        (size_t (*)(int64_t, int64_t))dlsym(lib, "_ZN3alp20emul_crt_sched_wordsEll");
    if (!words) return 3;
    const int order[4] = {0, 1, 0, 1};
    for (int i = 0; i < 4; ++i) {
        device = order[i];
        printf("%d ", clusters(words(256 * 1000, 256), 1000));
    }
    return 0;
}
"""


def test_clusters_of_each_device(alp, tmp_path):
    src, exe = tmp_path / "clusters.c", tmp_path / "clusters"
    src.write_text(PROGRAM)
    subprocess.run(["gcc", "-O1", "-rdynamic", "-o", str(exe), str(src), "-ldl"], check=True)
    r = subprocess.run([str(exe), alp.LIB_PATH], capture_output=True, text=True, timeout=120)
    if r.returncode == 3:
        pytest.fail("emul_crt_sched_words is not exported")
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["44", "30", "44", "30"]
