"""The line kernels' exchanges between the lanes of a warp, on the CPU (warp_emulation.h): the source
of the kernels is compiled for the host and run with the lanes of each warp taken in rising and in
falling order between two synchronisations.  A store that another lane's load of the stage before does
not wait for gives another result in one of the orders."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2309_12019_gb300", "csrc", "dgw_line_impl.cuh")
MAIN = r"""
template <class K> static int differ(K kernel, int nc, int order, int bc)
{
    const int cells = 8;
    std::vector<double> U[2];
    for (int up = 0; up < 2; ++up) {
        U[up].resize(nc * cells);
        for (int i = 0; i < nc * cells; ++i) U[up][i] = 1.0 + 0.3 * std::fmod(0.377 * (i + 1), 1.0);
        unsigned flag = 0;
        KParams A = {};
        A.h = A.two_h = 0.25; A.hh = 0.125; A.w_nbr = 0.01; A.eps_w = 1e-6; A.eps_s = 1e-12; A.q_one = 1;
        A.stab = STAB_WENO; A.nx = cells; A.E = cells; A.flag = &flag;
        for (int& b : A.bc) b = bc;
        LineSteps L = {};
        L.Uin = L.U = U[up].data(); L.nsteps = 2; L.order = order; L.stages = order == 4 ? 10 : order; L.cells = cells;
        for (int i = 0; i < 3; ++i) { L.cn[i] = 0.3 * i; L.ck[i] = 1.0 - 0.3 * i; L.cl[i] = 1e-3; }
        run_lanes(8 * cells, up == 1, [&] { kernel(A, L); });
    }
    return std::memcmp(U[0].data(), U[1].data(), U[0].size() * sizeof(double)) != 0;
}
int main()
{
    int bad = 0;
    for (int order : {2, 3, 4})
        for (int bc : {BC_PERIODIC, BC_REFLECT}) {
            bad += differ(line_wide_euler_kernel<DEG>, 3 * (DEG + 1), order, bc);
            bad += differ(line_wide_kernel<DEG, FLUX_BURGERS>, DEG + 1, order, bc);
        }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


@pytest.mark.parametrize("p", [1, 2, 3])
def test_lane_order_does_not_matter(p, tmp_path):
    with open(SRC) as fh:
        src = fh.read()
    src = src[:src.index("// Largest cluster of `fn`")]       # the kernels without their launches
    # the functions that hold machine instructions, which the header replaces
    src, n = re.subn(r"__device__ __forceinline__ \w+ (?:cluster_\w+|st_cluster)\([^)]*\)\s*\{.*?\}\n(?=\n|__device__)", "", src,
                     flags=re.S)
    assert n == 4 and "asm" not in src
    # (of a kernel that is not run here)
    src = src.replace("extern __shared__", "static").replace("smem_line[]", "smem_line[16]")
    f = tmp_path / "line.cpp"
    f.write_text('#include "warp_emulation.h"\n' + src + MAIN.replace("DEG", str(p)))
    exe = str(tmp_path / "line")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", HERE, str(f), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
