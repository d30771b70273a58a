"""The host half of the library over the stand-in runtime (host_api.py): what it plans, uploads and
launches."""
import ctypes

import numpy as np
import pytest

import host_api
from paper_2602_05017_gb300 import binding


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_api.load(str(tmp_path_factory.mktemp("host")))


# Longest line the pipelined sweep takes for 1 .. 32 substrates with one column per thread and a
# [T][T][S] table of carry weights, 227 KB of shared memory: (axis > 0, bytes per element).
LONGEST = {
    (0, 4): [1280, 1280, 1280, 1155, 1112, 1152, 992, 800, 1018, 906, 768, 704, 640, 608, 576, 544,
             448, 448, 448, 433, 416, 384, 384, 352, 352, 336, 320, 320, 297, 288, 288, 279],
    (0, 2): [1280, 1280, 1280, 1280, 1280, 1280, 1280, 1124, 1184, 1088, 992, 800, 752, 704, 672,
             624, 448, 448, 448, 448, 448, 448, 448, 416, 416, 384, 384, 362, 352, 352, 320, 320],
    (1, 4): [1408, 1404, 1270, 1152, 1070, 992, 864, 800, 762, 704, 672, 640, 608, 576, 558, 544,
             512, 500, 480, 452, 448, 428, 416, 416, 384, 384, 380, 352, 352, 352, 320, 320],
    (1, 2): [1408, 1408, 1408, 1408, 1408, 1344, 1220, 1120, 1040, 864, 816, 768, 736, 684, 640,
             624, 608, 576, 544, 512, 512, 480, 480, 448, 448, 416, 416, 384, 384, 384, 352, 352],
}


@pytest.mark.parametrize("esz", [4, 2])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_pipelined_lines_are_no_shorter(lib, axis, esz):
    out = (ctypes.c_int * 3)()
    unit = 16 // esz  # elements of a 16-byte row
    for ns, longest in enumerate(LONGEST[min(axis, 1), esz], 1):
        for n in {*range(1, longest, 7), *range(max(1, longest - 64), longest + 1)}:
            dims = [8, 8, 8]
            dims[axis] = n
            gp = -(-dims[0] * ns // unit) * unit
            assert lib.stand_in_pipe_shape(axis, *dims, ns, esz, gp, 0, 0, out), (n, ns)


@pytest.mark.parametrize("shape", [(8, 1000, 4, 9), (1272, 8, 4, 7), (8, 8, 448, 25)],
                         ids=lambda s: "x".join(map(str, s)))
def test_long_16_bit_lines_at_odd_substrate_counts(lib, shape):
    st, h = host_api.create(lib, *shape, "bf16")
    assert st == binding.OK
    assert host_api.describe(lib, h).count("pipe") == 3
    lib.biofvm_destroy(h)


@pytest.mark.parametrize("shape", [(4, 1256, 3, 3), (1072, 4, 4, 5), (4, 8, 1000, 7)],
                         ids=lambda s: "x".join(map(str, s)))
def test_long_fp32_lines_at_odd_substrate_counts(lib, shape):
    st, h = host_api.create(lib, *shape, "fp32")
    assert st == binding.OK
    assert host_api.describe(lib, h).count("pipe") == 3
    lib.biofvm_destroy(h)


@pytest.mark.parametrize("cw", [0, 16, 24, 32])
@pytest.mark.parametrize("chunk", [1, 8, 16, 20, 24, 32, 48, 64, 500])
def test_a_forced_tile_never_refuses_an_axis(lib, chunk, cw):
    out = (ctypes.c_int * 3)()
    for axis in range(3):
        for n, ns in ((40, 1), (400, 4), (1000, 2), (1100, 5)):
            dims = [8, 8, 8]
            dims[axis] = n
            assert lib.stand_in_pipe_shape(axis, *dims, ns, 4, dims[0] * ns, chunk, cw, out)
            if n == 40 and cw in (0, 32):  # fits: the capacity that holds the length
                caps = [16, 24] if axis == 0 else [16, 24, 48]
                assert out[:2] == [32, next((c for c in caps if c >= chunk), caps[-1])]


@pytest.mark.parametrize("chunk", ["32", "48"])
def test_16_bit_handles_under_a_forced_chunk(lib, chunk, monkeypatch):
    monkeypatch.setenv("BIOFVM_PIPE_CHUNK", chunk)
    st, h = host_api.create(lib, 64, 64, 64, 2, "fp16")
    assert st == binding.OK
    assert host_api.describe(lib, h) == "x=pipe/cw32/m24 y=pipe/cw32/m48 z=pipe/cw32/m48"
    lib.biofvm_destroy(h)


@pytest.mark.parametrize("grid", [(96, 96, 96, 2), (97, 95, 96, 1)], ids=["aligned", "padded"])
def test_a_batch_environments_own_step_takes_the_whole_gpu(lib, grid, monkeypatch):
    monkeypatch.setenv("BIOFVM_BATCH_MODE", "graph")
    st, h = host_api.create(lib, *grid, "fp32")
    st_b, b = host_api.create_batch(lib, [grid] * 12, "fp32")
    assert st == st_b == binding.OK
    env = ctypes.c_void_p()
    assert lib.biofvm_batch_env(b, 3, ctypes.byref(env)) == binding.OK
    seen = []
    for step, what in ((lib.biofvm_step, h), (lib.biofvm_step, env), (lib.biofvm_batch_step, b)):
        lib.stand_in_forget_launches()
        assert step(what, 1) == binding.OK
        seen.append([(r.grid, r.overlap) for r in host_api.pipe_launches(lib)[:3]])
    assert seen[1] == seen[0]
    assert all(batch[0] < alone[0] and not batch[1] for batch, alone in zip(seen[2], seen[0]))
    lib.biofvm_destroy(h)
    lib.biofvm_batch_destroy(b)


def test_a_failed_upload_leaves_no_sources_and_a_matching_map(lib):
    nvox, ns = 16 * 12 * 10, 2
    st, h = host_api.create(lib, 16, 12, 10, ns, "fp32")
    assert st == binding.OK

    def agents(n):
        rates = np.ones((n, ns))
        voxel = np.arange(n, dtype=np.int64) % nvox
        return lib.biofvm_set_sources(h, n, *(ctypes.c_void_p(a.ctypes.data) for a in (
            voxel, rates, rates, rates)), None)

    def adjoint():  # entries walked, entries of the map, largest entry, entries of the list
        field, saved = np.zeros(nvox * ns, np.float32), np.zeros(4 * nvox * ns, np.float32)
        grads = [np.zeros(4096) for _ in range(3)]
        ptr = [ctypes.c_void_p(a.ctypes.data) for a in (field, field, *grads, saved)]
        assert lib.biofvm_adjoint_step(h, *ptr) == binding.OK
        out = (ctypes.c_int64 * 4)()
        lib.stand_in_source_adjoint(out)
        return list(out)

    for n in (5, 700, 3):
        assert agents(n) == binding.OK
        assert adjoint() == [n * ns, adjoint()[1], n * ns - 1, n * ns] and adjoint()[1] >= n * ns
        graphs = lib.stand_in_graphs_made()
        assert lib.biofvm_step(h, 1) == binding.OK
        lib.stand_in_fail_allocation(0)
        assert agents(1500) == binding.ERR_OOM
        lib.stand_in_fail_allocation(-1)
        walked, held, largest, entries = adjoint()
        assert walked == 1500 * ns and held >= walked and largest == -1 and entries == 0
        assert lib.biofvm_step(h, 1) == binding.OK  # a new graph: the old one reads freed lists
        assert lib.stand_in_graphs_made() == graphs + 2
    lib.biofvm_destroy(h)


@pytest.mark.parametrize("steps", [1, 2, 3, 10])
@pytest.mark.parametrize("grid", [(41, 37, 29, 2), (64, 32, 16, 2)], ids=["padded", "aligned"])
def test_one_graph_a_call(lib, grid, steps):
    st, h = host_api.create(lib, *grid, "fp32")
    assert st == binding.OK
    graphs = lib.stand_in_graphs_made()
    for _ in range(3):
        assert lib.biofvm_step(h, steps) == binding.OK
    assert lib.stand_in_graphs_made() == graphs + 1
    lib.biofvm_destroy(h)


@pytest.mark.parametrize("grid, overlap", [((360, 360, 360, 1), 1), ((256, 256, 256, 4), 0)])
def test_overlapped_launches_up_to_200_megabytes(lib, grid, overlap):
    st, h = host_api.create(lib, *grid, "fp32")
    assert st == binding.OK
    lib.stand_in_forget_launches()
    assert lib.biofvm_step(h, 1) == binding.OK
    assert [r.overlap for r in host_api.pipe_launches(lib)] == [overlap] * 3
    lib.biofvm_destroy(h)
