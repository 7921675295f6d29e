"""host::resident_clusters on the CPU: host.cu compiled with stand-ins for the runtime's queries."""
import os
import subprocess

from paper_2303_11257_b200 import build as B

MAIN = """#include "%s"
#include <cstdio>
int asked;
static us::host::ClusterCount first, second;
int main() {
  auto ask = [](long kern, int cluster, us::host::ClusterCount& c) { printf("%%d ", us::host::resident_clusters((void*)kern, 640, 1000, cluster, c)); };
  ask(100, 2, first); ask(200, 2, second); ask(100, 4, first); ask(100, 2, first); ask(200, 2, second); ask(0, 2, first); ask(100, 1, first); ask(100, 9, first);
  printf("%%d", asked);
}
"""
# the number of clusters that fit is what the test gives as the kernel's address
STAND_INS = """extern int asked;
extern "C" {
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 148; return 0; }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaOccupancyMaxActiveClusters(int* n, const void* kern, const void*) { ++asked; *n = (int)(long)kern; return 0; }
}
"""


def test_the_count_of_resident_clusters_is_a_kernels_own(tmp_path):
    (tmp_path / "main.cu").write_text(MAIN % os.path.join(B.CSRC, "host.cu"))
    (tmp_path / "runtime.cpp").write_text(STAND_INS)
    exe = str(tmp_path / "main")
    subprocess.run([B._nvcc(), "-std=c++17", "-cudart", "shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", exe, str(tmp_path / "main.cu"),
                    str(tmp_path / "runtime.cpp")], check=True, capture_output=True, text=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split() == ["100", "200", "100", "100", "200", "100", "148", "-1", "3"]
