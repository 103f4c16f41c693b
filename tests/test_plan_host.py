"""The launch plan (csrc/plan.h) on the CPU: what each warp's shared slab holds and
which launch shape a context takes."""
import os
import subprocess

import pytest

from paper_2603_03639_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "%s"
// N K chi M P operator warps ctas_per_sm free_GB -> warps, CTA slots, slab elements,
// resident CTAs per SM by shared memory, GB
int main(int argc, char** argv) {
  tnrc_problem pb{};
  pb.struct_size = sizeof(pb);
  pb.n_sites = atoi(argv[1]);
  pb.n_slices = atoi(argv[2]);
  pb.chi_max = atoi(argv[3]);
  pb.n_samples = atoi(argv[4]);
  pb.n_inputs = atoi(argv[5]);
  pb.operator_form = atoi(argv[6]);
  pb.warps_per_cta = atoi(argv[7]);
  pb.ctas_per_sm = atoi(argv[8]);
  pb.n_controls = 2;
  pb.dt = 0.05;
  const double free_gb = atof(argv[9]);
  tnrc_host::Plan P;
  if (!tnrc_host::make_plan(&pb, 152, (size_t)(free_gb * 1e9), P, free_gb > 0)) {
    printf("refused\n");
    return 0;
  }
  printf("%%d %%d %%d %%.4f\n", P.warps, P.grid, P.slab_elems, P.total / 1e9);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(PROGRAM % os.path.join(build.CSRC, "plan.h"))
    exe = str(d / "plan")
    subprocess.run([build.nvcc(), "-std=c++17", "-o", exe, str(d / "plan.cu"), "-L", build.LIBDIR, "-ltnrc", "-Xlinker",
                    "-rpath=" + build.LIBDIR], check=True)
    env = {k: v for k, v in os.environ.items() if not k.startswith("TNRC_")}

    def run(N, K, chi, M, P=1, operator=0, warps=0, ctas=0, free=0.0):
        out = subprocess.run([exe] + [str(x) for x in (N, K, chi, M, P, operator, warps, ctas, free)],
                             capture_output=True, text=True, check=True, env=env).stdout.split()
        return None if out == ["refused"] else dict(zip(("warps", "grid", "slab", "gb"),
                                                        (int(out[0]), int(out[1]), int(out[2]), float(out[3]))))
    return run


@pytest.mark.parametrize("operator", [0, 1])
@pytest.mark.parametrize("N", [2, 3, 5, 8, 32, 33])
@pytest.mark.parametrize("shape", [(8, 1), (4, 2), (2, 1), (2, 4), (4, 4)])
def test_slab_holds_the_updates_that_the_shared_memory_can(plan, N, operator, shape):
    """The largest update (theta, R^dagger, pivot column and Phi), two of them from 33
    sites on, and the gradient's product and intermediates fit the slab, or it is all
    that the SM leaves to a warp: 220 KB shared by its CTAs, less 4 KB of arrays a warp
    and 1 KB."""
    if operator and shape[0] * shape[1] > 8:
        pytest.skip("operators run up to 8 warps an SM")
    d = 4 if operator else 2
    left = (220 * 1024 // shape[1] - shape[0] * 4096 - 1024) // shape[0] // 16 // 32 * 32
    for chi in (1, 2, 3, 4, 5, 7, 8, 9, 13, 16, 19, 20, 32):
        D = [min(chi, d ** min(i, 6), d ** min(N - i, 6)) for i in range(N + 1)]
        need = 0
        for b in range(N - 1):
            m, n = d * D[b], d * D[b + 2]
            upd = 2 * m * n + min(m, n) * (n | 1) + m
            need = max(need, 2 * upd if N >= 33 else upd, 2 * m * n + D[b] * d * D[b + 1] + D[b] * d * d * D[b + 2])
        p = plan(N, 10, chi, 8, operator=operator, warps=shape[0], ctas=shape[1])
        assert p["slab"] == max(256, min(need, left))


@pytest.mark.parametrize("N,K,chi,operator", [(50, 16, 32, 0), (30, 16, 64, 0), (12, 12, 32, 0), (4, 8, 16, 1)])
def test_two_ctas_per_sm_from_one_trajectory_more_than_sms(plan, N, K, chi, operator):
    for T, shape in ((1, (8, 1)), (152, (8, 152)), (153, (4, 153)), (304, (4, 304)), (1000, (4, 304))):
        p = plan(N, K, chi, T, operator=operator)
        assert (p["warps"], p["grid"]) == shape


def test_one_cta_per_sm_where_two_take_tens_of_gb(plan):
    p = plan(50, 100, 64, 256, 8)
    assert (p["warps"], p["grid"]) == (8, 152)
    assert plan(50, 100, 64, 256, 8, warps=4, ctas=2)["grid"] == 304   # unless asked for


def test_operators_that_need_half_an_sm_keep_one_cta(plan):
    assert plan(8, 8, 16, 300, operator=1)["warps"] == 8


def test_two_ctas_per_sm_only_where_their_regions_fit(plan):
    """Where the free memory limits the CTAs, one CTA with all warps per SM takes the
    regions that fit; a problem that fits so is not refused."""
    args = (50, 64, 32, 128, 8)
    full = plan(*args)
    assert (full["warps"], full["grid"]) == (4, 304)
    one = plan(*args, warps=8, ctas=1)
    assert one["grid"] == 152 and one["gb"] < 0.6 * full["gb"]
    for free, warps, grid in ((1.3 * full["gb"], 4, 304), (1.1 * full["gb"], 8, 152), (1.3 * one["gb"], 8, 152)):
        p = plan(*args, free=free)
        assert (p["warps"], p["grid"]) == (warps, grid)
    few = plan(*args, free=0.7 * one["gb"])
    assert few["warps"] == 8 and 0 < few["grid"] < 152


def test_a_context_of_four_warps_is_kept_where_eight_do_not_fit(plan):
    """Short chains at chi = 64: a region is mostly its warps' scratch (1.2 MB each)."""
    args = (10, 4, 64, 160)
    fixed = plan(*args)["gb"] - 160 * (plan(*args)["gb"] - plan(*args, warps=4, ctas=1)["gb"]) / 8.0   # without regions
    four = (plan(*args)["gb"] - fixed) / 160
    eight = (plan(*args, warps=8, ctas=1)["gb"] - fixed) / 152
    assert eight > 1.3 * four
    p = plan(*args, free=(fixed + 0.5 * (four + eight)) / 0.85)
    assert p is not None and p["warps"] == 4 and p["grid"] == 1
