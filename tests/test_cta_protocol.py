"""What the warps of the tcgen05 kernels tell each other, in any order of the warps and with waits that expire: the kernels' own sources on
the host, a warp a fiber (cta_emulation.h).  No GPU: a CTA whose wait has expired is not something to bring about on one."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2606_08804_b200", "csrc")

MAIN = r"""
using namespace qd;
static std::vector<float> F(1 << 22);                    // stands for every buffer
static float* f() { return F.data(); }
static bf16* h() { return reinterpret_cast<bf16*>(F.data()); }
static unsigned* u() { return reinterpret_cast<unsigned*>(F.data()); }
static CUtensorMap box(long bytes) { CUtensorMap m{}; m.opaque[0] = (uint64_t)bytes; return m; }
%s
int main(int argc, char** argv) {
    const std::string name = argv[1];
    const int runs = atoi(argv[2]);
    const double expire = atof(argv[3]), lose = atof(argv[4]);
    int aborted = 0;
    for (int i = 0; i < runs; ++i) {
        emu::Scenario s{(unsigned)i, expire, lose, true};
        const std::string e = one(name, s, i);
        if (!e.empty()) { printf("run %%d: %%s\n", i, e.c_str()); return 1; }
        aborted += emu::c_expired;
        if (lose == 0 && expire == 0 && emu::c_expired) { printf("run %%d: a wait expired\n", i); return 1; }
    }
    if (expire > 0 && aborted < runs / 4) { printf("waits expired in %%d of %%d runs only\n", aborted, runs); return 1; }
    printf("ok %%d\n", aborted);
}
"""

FWD = r"""
static std::string one(const std::string& name, const emu::Scenario& s, int i) {
    const int N = 1 + i % 8;
    if (name == "prep") {
        PrepParams p{};
        p.T = p.Tp = 64 * N; p.H = 1; p.N = p.Ns = N; p.BH = 1;
        p.beta = p.alpha = p.lam = h(); p.g = f(); p.Qg = h(); p.Mt = h(); p.rqk = f(); p.status = u();
        const auto kern = i & 1 ? k_tc_prep<true, true> : k_tc_prep<false, false>;
        return emu::run(s, kPrepThreads, dim3(i % N), dim3(N), [&] { kern(box(8192), box(8192), box(8192), box(0), box(0), box(0), p); });
    }
    ChainParams p{};
    p.T = p.Tp = 64 * N; p.H = 1; p.N = p.Ns = N; p.g = f(); p.hT = f(); p.o = h(); p.scaled = i & 1; p.rk = f(); p.status = u();
    if (name == "half") {
        const auto kern = i & 8 ? k_tc_chain_fwd_half<true> : k_tc_chain_fwd_half<false>;
        return emu::run(s, kHalfThreads, dim3(i & 1), dim3(2), [&] { kern(box(16384), box(8192), box(8192), box(8192), box(8192), box(0), box(0), p); });
    }
    const auto kern = i & 8 ? k_tc_chain_fwd<true> : k_tc_chain_fwd<false>;
    return emu::run(s, kChainThreads, dim3(0), dim3(1), [&] { kern(box(16384), box(16384), box(8192), box(8192), box(8192), box(0), box(0), box(0), p); });
}
"""

BWD = r"""
static std::string one(const std::string& name, const emu::Scenario& s, int i) {
    const int N = 1 + i % 8;
    if (name == "chunk") {
        ChunkBwdParams p{};
        p.T = p.Tp = 64 * N; p.H = 1; p.N = p.Ns = p.total = N; p.BH = 1; p.group = 1;
        p.beta = p.alpha = p.lam = h(); p.g = f(); p.dbeta = p.dalpha = p.dlam = f(); p.rqk = f(); p.status = u(); p.next = u() + 1;
        *p.next = 0;
        F[0] = F[1] = 0;
        ChunkBwdMaps m{};
        m.Q = m.K = m.V = m.dO = m.Mt = m.P = box(8192);
        m.Dt = m.dDt = m.Hs = m.dHs = box(16384);
        const auto kern = i & 8 ? k_tc_chunk_bwd<true, true, true> : i & 16 ? k_tc_chunk_bwd<false, false, false> : k_tc_chunk_bwd<true, true, false>;
        return emu::run(s, kBwdThreads, dim3(0), dim3(1), [&] { kern(m, p); });
    }
    ChainBwdParams p{};
    p.Tp = 64 * N; p.H = 1; p.N = p.Ns = N; p.rk = f(); p.g = f(); p.dhT = f(); p.dh0 = f(); p.status = u(); p.next = u() + 1; p.dhT_early = i & 1;
    const auto kern = i & 8 ? k_tc_chain_bwd<D> : k_tc_chain_bwd<D / 2>;
    return emu::run(s, kChainThreads, dim3(0), dim3(1), [&] { kern(box(16384), box(8192), box(8192), box(8192), box(8192), box(0), box(0), p); });
}
"""


def _source(name):
    src = open(os.path.join(CSRC, name)).read()
    src = src[:src.index("\ntemplate <class K>\ncudaError_t set_smem")] + "\n}\n}\n"
    src = re.sub(r'#include "(sm100|tf32)\.cuh"', "", src)
    src = re.sub(r"extern __shared__ [^;]*;", "unsigned char* const smem_raw = emu::smem;", src)
    src = src.replace("__shared__ ", "static ").replace("__grid_constant__ ", "")
    src = re.sub(r"__launch_bounds__\([^)]*\)", "", src)
    src = re.sub(r'asm volatile\("bar\.sync (\d), %0;" ::"n"\((\w+)\) : "memory"\);', r"sm100::nb_sync(\1, \2);", src)
    src = re.sub(r'asm volatile\("bar\.sync (\d), (\d+);" ::: "memory"\);', r"sm100::nb_sync(\1, \2);", src)
    src = re.sub(r'asm volatile\("bar\.sync %0, %1;" ::"r"\((\w+)\), "r"\((\w+)\) : "memory"\);', r"sm100::nb_sync(\1, \2);", src)
    assert "asm " not in src
    return '#include "cta_emulation.h"\n' + src


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    """The two files' kernels as host programs, compiled when first asked for."""
    out = {}

    def get(name):
        if name not in out:
            d = tmp_path_factory.mktemp("emu")
            cpp, exe = str(d / "cta.cpp"), str(d / "cta")
            with open(cpp, "w") as fh:
                fh.write(_source(name) + MAIN % (FWD if name == "tc_fwd.cu" else BWD))
            r = subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-Wno-psabi", "-I", HERE, "-I", CSRC, "-I", "/usr/local/cuda/include", cpp,
                                "-o", exe], capture_output=True, text=True)
            assert r.returncode == 0, r.stderr[:4000]
            out[name] = exe
        return out[name]
    return get


ALL = [("tc_fwd.cu", "prep"), ("tc_fwd.cu", "full"), ("tc_fwd.cu", "half"), ("tc_bwd.cu", "chain"), ("tc_bwd.cu", "chunk")]


def _run(exe, kernel, runs, expire, lose):
    r = subprocess.run([exe, kernel, str(runs), str(expire), str(lose)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("name,kernel", ALL)
def test_any_order_of_warps(programs, name, kernel):
    """No wait expires, and the CTA leaves with everything done."""
    _run(programs(name), kernel, 100, 0, 0)


@pytest.mark.parametrize("name,kernel", ALL)
@pytest.mark.parametrize("expire,lose", [(0.0005, 0), (0.05, 0), (0.005, 0.02)], ids=["rare", "early", "lost load"])
def test_expired_waits(programs, name, kernel, expire, lose):
    """Waits expire at any place, copies are lost: the kernel comes to its end all the same, and leaves as cleanly."""
    _run(programs(name), kernel, 200, expire, lose)
