"""A resident team whose launch the device refuses is not run, and the caller is
told so that the solve streams (host only: csrc/resident.cu with the CUDA calls
replaced by fakes that refuse)."""
import os
import subprocess

from paper_2106_07616_gb300 import _build

MAIN = r"""
#include "resident.cuh"
#include "krylov.cuh"

static cudaError_t attr_rc, launch_rc;
static int launched, cluster, cooperative;
template <typename F>
static cudaError_t fake_attr(F *, cudaFuncAttribute, int) { return attr_rc; }
static cudaError_t fake_launch(const cudaLaunchConfig_t *c, const void *, void **) {
  ++launched;
  cluster = cooperative = 0;
  if (c->attrs[0].id == cudaLaunchAttributeClusterDimension)
    cluster = (int)c->attrs[0].val.clusterDim.x;
  else
    cooperative = c->attrs[0].val.cooperative;
  return launch_rc;
}
#define cudaFuncSetAttribute fake_attr
#define cudaLaunchKernelExC fake_launch
#include "resident.cu"
namespace rbffd {
void set_error(const char *, ...) {}
}  // namespace rbffd
using namespace rbffd;

int main() {
  rbffd_ctx ctx;
  for (int one_cluster = 0; one_cluster < 2; ++one_cluster)
    for (int refuse = 0; refuse < 3; ++refuse) {
      ResPlan p;
      p.nb = one_cluster ? 16 : 152;
      p.cluster = one_cluster;
      attr_rc = refuse == 1 ? cudaErrorInvalidValue : cudaSuccess;
      launch_rc = refuse == 2 ? cudaErrorCooperativeLaunchTooLarge : cudaSuccess;
      launched = 0;
      const int64_t before = ctx.launches;
      const bool ran = res_launch(&ctx, p, (const void *)main, nullptr, 1000);
      printf("%d%d%d:%d:%d ", ran, (int)(ctx.launches - before), launched, cluster, cooperative);
    }
}
"""


def test_refused_launches_are_not_run(tmp_path):
    (tmp_path / "refused.cu").write_text(MAIN)
    exe = str(tmp_path / "refused")
    subprocess.run(["nvcc", *_build.ARCH, "-std=c++17", "-I", os.path.join(_build.HERE, "csrc"),
                    "-I", _build.INCLUDE, "-o", exe, str(tmp_path / "refused.cu")], check=True,
                   capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    # ran, counted, launched: cluster size: cooperative
    assert out == ["111:0:1", "000:0:1", "001:0:1", "111:16:0", "000:16:0", "001:16:0"]
