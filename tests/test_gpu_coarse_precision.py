"""The coarsest solve in clusters is no further from 64 bits than the solve with one block per right-hand side and FP64
sums that it took the place of: V-cycles against the FP64 oracle, the bounds are that solve's errors on the same
inputs.  And its sums over lanes, on their own, keep what FP64 keeps."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import multigrid as MG  # noqa: E402
from paper_2405_17696_gb300 import build as B  # noqa: E402
from paper_2405_17696_gb300 import media  # noqa: E402

SUMS = """
#include "reduce.cuh"
// 8 values per lane of one warp -> their sums as doubles; then one complex value per lane, summed over groups
__global__ void sums(const float* v, double* out8, const float2* g, int wide, double2* outg) {
    const int lane = threadIdx.x;
    float a[8];
    for (int k = 0; k < 8; ++k) a[k] = v[8 * lane + k];
    const helm::tf s = helm::tf_warp_sum8(a, lane);
    if ((lane & 3) == 0) out8[lane >> 2] = helm::tf_double(s);
    const float2 z = make_float2(0.f, 0.f);
    const helm::tf2 t = helm::tf2_group_sum({g[lane], z, z}, wide);
    outg[lane] = make_double2(helm::tf_double(helm::first_of(t)), helm::tf_double(helm::second_of(t)));
}
extern "C" int run(const float* v, double* out8, const float2* g, int wide, double2* outg) {
    sums<<<1, 32>>>(v, out8, g, wide, outg);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    from paper_2405_17696_gb300 import native as n
    return n


@pytest.mark.parametrize("nx,nz,levels,k,h,bound", [
    (64, 32, 2, 10, 20.0, 2.2375e-7),
    (64, 32, 2, 16, 5.0, 3.4634e-7),
    (128, 64, 3, 10, 10.0, 2.6037e-7),
])
def test_vcycle_error_no_larger_than_with_fp64_sums(native, nx, nz, levels, k, h, bound):
    dev = torch.device("cuda:0")
    kap, gam = media.kappa_of(media.layered_velocity(nx, nz, seed=5)), media.abl_gamma(nx, nz, 8)
    om, nb = np.asarray([2 * np.pi * 4.0], np.float32), 16
    f = media.complex_normal((nb, nz, nx), 7)
    opts = native.helm_default_opts(mg_levels=levels, coarse_iters=k, max_rhs=nb, restart=1,
                                    stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(torch.from_numpy(kap).to(dev), torch.from_numpy(gam).to(dev), nx, nz, h, h,
                            torch.from_numpy(om).to(dev), opts=opts)
    try:
        u = torch.empty((nb, nz, nx), dtype=torch.complex64, device=dev)
        native.helm_vcycle(ctx, torch.from_numpy(f).to(dev), None, u, nb)
        got = u.cpu().numpy()
    finally:
        native.helm_destroy(ctx)
    pc = MG.VCyclePreconditioner(kap.astype(np.float64), gam.astype(np.float64), float(om[0]), h, h,
                                 MG.VCycleParams(levels=levels, coarse_iters=k, jacobi_w=float(np.float32(0.8))))
    ref = [pc(x.astype(np.complex128)) for x in f]
    err = [np.linalg.norm(g - r) / np.linalg.norm(r) for g, r in zip(got, ref)]
    assert math.sqrt(np.mean(np.square(err))) <= bound


@pytest.mark.parametrize("wide", [1, 2, 8, 32])
def test_lane_sums_are_exact_to_fp64(native, tmp_path, wide):
    src, lib = tmp_path / "sums.cu", tmp_path / "sums.so"
    src.write_text(SUMS)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(lib)], check=True)
    run = ctypes.CDLL(os.fspath(lib)).run
    rng = np.random.default_rng(wide)
    # 40 binary orders of magnitude, and large values that cancel but for the last one's part
    v = (rng.normal(size=(32, 8)) * 2.0 ** rng.integers(-20, 20, (32, 8))).astype(np.float32)
    v[1::2, 4:] = -v[0::2, 4:]
    v[31, 4:] += np.abs(v[31, 4:]) * np.float32(1e-3)
    g = (rng.normal(size=(32, 2)) * 2.0 ** rng.integers(-20, 20, (32, 2))).astype(np.float32)
    dv, dg = torch.from_numpy(v).cuda(), torch.from_numpy(g).cuda()
    o8, og = torch.zeros(8, dtype=torch.float64).cuda(), torch.zeros((32, 2), dtype=torch.float64).cuda()
    assert run(*(ctypes.c_void_p(x.data_ptr()) for x in (dv, o8, dg)), wide, ctypes.c_void_p(og.data_ptr())) == 0

    def check(got, terms):
        # three terms drop what lies 2^-66 below the terms; adding them up in FP64 rounds twice
        t = [float(x) for x in terms]
        assert abs(got - math.fsum(t)) <= 2.0 ** -66 * sum(map(abs, t)) + 2.0 ** -52 * abs(math.fsum(t))

    for k in range(8):
        check(float(o8[k]), v[:, k])
    for lane in range(32):
        for part in range(2):
            check(float(og[lane, part]), g[lane // wide * wide:][:wide, part])
