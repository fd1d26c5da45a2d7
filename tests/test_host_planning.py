"""Host code of the library over a stand-in for the CUDA runtime (fake_cudart.cpp): which kernels a call launches and how
large, also where the driver refuses something.  No device."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2506_12040_b200 import build
from paper_2506_12040_b200.binding import BtcLinearProblem, BtcTransform
from util import EPILOGUE_SHAPES

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("fake") / "libbtc_fake.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-isystem", "/usr/local/cuda/include",
                           os.path.join(HERE, "fake_cudart.cpp"), *build.objects(), "-o", lib])
    L = ctypes.CDLL(lib)
    L.fake_name.restype = ctypes.c_char_p
    L.fake_coop_args.restype = ctypes.c_void_p
    L.btc_codebook_kmeans_workspace_bytes.restype = ctypes.c_size_t
    L.fake_reset.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    return L


def _launches(L):
    return [(L.fake_name(i).decode(), L.fake_grid(i)) for i in range(L.fake_count())]


def test_a_refused_layer_of_a_batch_does_not_launch_the_others_twice(fake):
    """Two layers of different forms, so two launches; the driver refuses the second one's index matrix: the first layer
    runs once, the second on the kernel that needs no description."""
    P = (BtcLinearProblem * 2)()
    for case, kernels in enumerate((["gemv_kernel", "gemv_kernel"], ["gemv_kernel", "decode"])):
        for i, M in enumerate((1, 4)):               # (matrices of their own: descriptions are kept by address)
            base = 0x100000 * (2 * case + i + 1)
            P[i] = BtcLinearProblem(base, base + 0x10000, base + 0x20000, base + 0x30000, None, base + 0x40000, 0, 2, M, 64, 256, 16, 256, 0, 0, 0)
        fake.fake_reset(148, 0, 0, P[1].idx if case else None)
        assert fake.btc_linear_gemv_batch(P, 2, None) == 0
        got = [n for n, _ in _launches(fake)]
        assert len(got) == 2 and all(k in n for k, n in zip(kernels, got)), got


@pytest.mark.parametrize("N,K,M,split", [(300, 4096, 16, True), (200, 11008, 9, True), (1000, 5120, 100, True), (640, 8192, 300, True),
                                         (4096, 11008, 77, True), (11008, 4096, 2048, False)])
def test_few_tiles_and_a_long_k_share_it_in_a_cluster(fake, N, K, M, split):
    """Also from the entry point without a workspace."""
    p = ctypes.c_void_p
    shape = (M, N, K, 16, 8192)
    for call, scratch in ((fake.btc_linear_gemm, (p(0x6000), ctypes.c_size_t(-(-4 * M // 256) * 256))), (fake.btc_linear_gemm_static_scratch, ())):
        fake.fake_reset(148, 0, 0, None)
        assert call(p(0x1000), 1, p(0x2000), p(0x3000), p(0x4000), None, None, p(0x5000), 2, *shape, *scratch, None) == 0
        (name, _), = _launches(fake)
        assert "gemm_ts_kernel" in name and (fake.fake_cluster(0) > 1) == split


@pytest.mark.parametrize("M,N,K,tile", EPILOGUE_SHAPES)
def test_tiles_of_the_epilogue_shapes(fake, M, N, K, tile):
    """The parity test of the results at the edges of tiles meets both forms of the kernel."""
    p = ctypes.c_void_p
    fake.fake_reset(148, 0, 0, None)
    assert fake.btc_linear_gemm(p(0x1000), 1, p(0x2000), p(0x3000), p(0x4000), None, None, p(0x5000), 2, M, N, K, 16, 500, p(0x6000),
                                ctypes.c_size_t(-(-4 * M // 256) * 256), None) == 0
    (name, grid), = _launches(fake)
    assert f"gemm_ts_kernelILi{256 if tile > 128 else 128}E" in name and fake.fake_cluster(0) == 1
    assert grid == -(-N // 128) * -(-M // tile) and fake.fake_smem(0) == (4 if tile > 128 else 8) * tile * 128 + 1024 + 32768 + 2000 + 14 * 8 + 16


def test_registers_of_the_tensor_core_path(tmp_path):
    """No form spills, and a CTA of the row sums (256 threads) fits the registers that one of 640 threads with x tiles above 128
    rows leaves of the SM's 65536: they run side by side where a mean term follows."""
    out = subprocess.check_output([build._nvcc(), *build.NVCC_FLAGS, "-Xptxas=-v", "-I", build.INCLUDE, "-I", build.CSRC, "-c",
                                   os.path.join(build.CSRC, "gemm_tcgen05.cu"), "-o", str(tmp_path / "gemm.o")], stderr=subprocess.STDOUT, text=True)
    found = re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers", out, re.S)
    regs = {name: -(-int(used) // 8) * 8 for name, _, _, used in found}
    wide = [r for name, r in regs.items() if re.search("gemm_ts_kernelILi256ELi4ELi1ELb0E", name)]
    sums, = [r for name, r in regs.items() if "rowsum_kernel" in name]
    assert len(wide) == 9 and max(wide) * 640 + sums * 256 <= 65536, (wide, sums)
    assert not [f for f in found if f[1] != "0" or f[2] != "0"]


@pytest.mark.parametrize("sms", [148, 64, 16, 4])
def test_launches_follow_the_sms_of_the_device(fake, sms):
    """One round of CTAs where a kernel takes its work in turn; tiles that fill the device many times are not split."""
    p = ctypes.c_void_p
    fake.fake_reset(sms, 0, 0, None)
    P = (BtcLinearProblem * 1)()
    for M in (1, 8):
        P[0] = BtcLinearProblem(0x1000, 0x10000 + M * 4096, 0x20000, 0x30000, None, 0x40000, 0, 2, M, 11008, 4096, 16, 8192, 0, 0, 0)
        assert fake.btc_linear_gemv_batch(P, 1, None) == 0
    T = BtcTransform(0x1000, 0x2000, 0x3000, 64, 64)
    for M in (1, 2048):
        assert fake.btc_activation_transform(p(0x4000), 0, ctypes.byref(T), p(0x50000), 0, M, 4096, None) == 0
    one, eight, row, rows = [g for _, g in _launches(fake)]
    assert sms < one <= 2 * sms and eight == sms and row == 8 and rows == sms
    fake.fake_reset(sms, 0, 0, None)
    assert fake.btc_linear_gemm(p(0x1000), 1, p(0x2000), p(0x3000), p(0x4000), None, None, p(0x5000), 2, 16, 1024, 8192, 16, 8192,
                                p(0x6000), ctypes.c_size_t(256), None) == 0
    (name, grid), = _launches(fake)
    assert "gemm_ts_kernel" in name and grid == 8 * fake.fake_cluster(0) and (fake.fake_cluster(0) > 1) == (sms > 16)


@pytest.mark.parametrize("M,k1,k2,kernel", [(1, 64, 64, "few"), (8, 17, 64, "few"), (3, 128, 128, "few"), (8, 65, 128, "few"), (8, 16, 64, ""), (1, 129, 64, ""),
                                            (8, 64, 80, ""), (9, 64, 64, "mma")])
def test_transform_of_a_few_rows_shares_no_sm(fake, M, k1, k2, kernel):
    """No two CTAs fit an SM (228 KB of shared memory, 1 KB of it per CTA taken by the system): as many as there are together would
    go to the SMs that a layer in front leaves first, and keep the layer behind from them."""
    T = BtcTransform(0x1000, 0x2000, 0x3000, k1, k2)
    fake.fake_reset(148, 0, 0, None)
    assert fake.btc_activation_transform(ctypes.c_void_p(0x4000), 0, ctypes.byref(T), ctypes.c_void_p(0x50000), 0, M, k1 * k2, None) == 0
    (name, grid), = _launches(fake)
    assert ("transform_few_kernel" in name) == (kernel == "few") and ("transform_mma_kernel" in name) == (kernel == "mma")
    if kernel == "few":
        assert grid == M * k2 // 8 and 2 * (fake.fake_smem(0) + 1024) > 228 * 1024


class KmArgs(ctypes.Structure):
    _fields_ = ([("vecs", ctypes.c_void_p), ("n", ctypes.c_size_t)] + [(k, ctypes.c_int) for k in ("v", "Kc", "max_iter")]
                + [(f"p{i}", ctypes.c_void_p) for i in range(12)] + [(k, ctypes.c_int) for k in ("words", "fields", "parts")])


def _kmeans(L, n, v, Kc=256):
    """Launches the construction; returns the grid and the arguments of the kernel."""
    p = ctypes.c_void_p
    rc = L.btc_codebook_kmeans(p(0x1000), ctypes.c_size_t(n), v, Kc, 5, p(0x2000), p(0x3000), p(0x4000), p(0x10000),
                               L.btc_codebook_kmeans_workspace_bytes(v, Kc), None)
    assert rc == 0
    (name, grid), = _launches(L)
    assert "km_kernel" in name
    return grid, KmArgs.from_address(L.fake_coop_args())


@pytest.mark.parametrize("v", [1, 13, 16, 20])
@pytest.mark.parametrize("n", [1, 3000, 1 << 20, (1 << 31) - 1])
@pytest.mark.parametrize("sms", [1, 2, 18, 35, 148, 300])
def test_codebook_construction_fits_its_tables_on_any_number_of_sms(fake, sms, n, v):
    """A part of the 2^v patterns: its frequencies, and as many places for those past the last bin, beside 2049 bins and twice 2048 words for
    the ranks in shared memory, its counts in 16 bits, a column of the 256 per bin; every pattern in one part, every CTA one
    part or more."""
    fake.fake_reset(sms, 0, 0, None)
    grid, a = _kmeans(fake, n, v)
    assert (a.n, a.v, a.fields) == (n, v, 3 if n < 1 << 21 else 2)
    per = -(-(1 << v) // a.parts)
    assert 1 <= grid <= min(sms, 256) and grid <= a.parts <= 256
    assert (2049 + 2 * 2048 + 2 * per) * 4 <= fake.fake_smem(0) and per < 1 << 16


@pytest.mark.parametrize("of_stream,most,grid", [(0, 0, 148), (16, 0, 16), (200, 0, 148), (0, 20, None), (64, 1, 1)])
def test_codebook_construction_takes_the_sms_it_is_given(fake, of_stream, most, grid):
    """A cooperative launch of a CTA per SM: those of the stream's green context, and where the launch is refused as too large
    all the same, as many as are let in (an eighth fewer each time)."""
    fake.fake_reset(148, of_stream, most, None)
    got, a = _kmeans(fake, 1 << 20, 20)
    assert got == grid or (grid is None and 7 * most // 8 <= got <= most), got
    assert (fake.fake_refused() > 0) == (most > 0) and a.parts == max(got, 128)


@pytest.mark.parametrize("n,v,Kc,copies", [(1 << 20, 16, 8192, False), (1 << 20, 16, 512, True), (1 << 20, 16, 513, False), (65535, 16, 512, False), (127, 12, 1, False), (128, 12, 1, True)])
def test_codebook_construction_keeps_copies_only_where_patterns_can_crowd(fake, n, v, Kc, copies):
    """128 patterns or more per centroid at most: there are no more of them than vectors, nor than 2^v."""
    fake.fake_reset(148, 0, 0, None)
    _kmeans(fake, n, v, Kc)
    assert f"km_kernelILb{int(copies)}E" in _launches(fake)[0][0]
