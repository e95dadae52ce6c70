"""The marching form (every step of an advance in one launch) against the CPU
oracle, bit for bit: tile and region edges, odd and tiny grids, step counts
around a phase, and the FP64 heat's integer arithmetic on the values where it
could differ from the FP64 operations."""
import numpy as np
import pytest

from paper_1602_07558_gb300 import inputs
from paper_1602_07558_gb300.swept2d import Swept2D, SweptBatch

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


def swept(op, u0, nsteps, tile, params, dtype=None):
    ny, nx = u0.shape[-2:]
    with Swept2D(nx, ny, op=op, tile=tile, params=params, dtype=dtype) as s:
        s.set_state(np.ascontiguousarray(u0.reshape(s.shape)))
        s.advance(nsteps)
        return s.get_state()


def field(kind, nx, ny):
    rng = np.random.default_rng(nx + 3 * ny)
    smooth = inputs.smooth_field(nx, ny, seed=2)
    smooth = smooth / np.abs(smooth).max()
    return {
        "one_binade": 1.5 + 0.2 * smooth,
        "binades": 3.0 + 2.9 * smooth,                 # 0.1 .. 5.9: six binades
        "negative": -2.0 - 0.5 * smooth,
        "crossing": smooth,
        "noise": rng.random((ny, nx)),
        "mixed_sign_noise": rng.standard_normal((ny, nx)),
        "ties": 1.0 + rng.integers(0, 2 ** 20, (ny, nx)) * 2.0 ** -52,
        "few_bits": 1.0 + rng.integers(0, 8, (ny, nx)) / 8.0,
        "powers": 2.0 ** rng.integers(-3, 3, (ny, nx)),
        "constant": np.full((ny, nx), 1.0),
        "zeros": np.zeros((ny, nx)),
        "tiny": (1.0 + 0.3 * smooth) * 2.0 ** -1060,   # below the normal numbers
        "smallest_normal": (1.0 + 0.3 * smooth) * 2.0 ** -1021,
        "huge": (1.0 + 0.3 * smooth) * 2.0 ** 1019,
    }[kind]


@pytest.mark.parametrize("r", [0.2, 0.125, 0.1875, 0.2499999, 0.25, 0.1, 0.0, -0.05])
@pytest.mark.parametrize("kind", ["one_binade", "binades", "negative", "crossing", "noise",
                                  "mixed_sign_noise", "ties", "few_bits", "powers", "constant",
                                  "zeros", "tiny", "smallest_normal", "huge"])
def test_fp64_heat_integer_arithmetic_is_bitwise(oracle_lib, kind, r):
    u0 = field(kind, 96, 64)
    with np.errstate(all="ignore"):
        ref = oracle_lib.heat(u0, r, 21)
    assert np.array_equal(swept("heat", u0, 21, 32, (r,))[0], ref, equal_nan=True)


def test_fp64_heat_keeps_infinities_and_nans_local(oracle_lib):
    u0 = field("one_binade", 128, 96)
    u0[5, 7], u0[60, 100] = np.inf, np.nan
    ref = oracle_lib.heat(u0, 0.2, 9)
    assert np.array_equal(swept("heat", u0, 9, 32, (0.2,))[0], ref, equal_nan=True)


# grids that take each of the shapes, with one tile, several, and sides smaller than the ring
@pytest.mark.parametrize("nx,ny,tile,nsteps", [
    (4, 4, 4, 9), (8, 200, 4, 11), (200, 8, 4, 11), (30, 30, 6, 7),
    (64, 48, 16, 1), (64, 48, 16, 2), (64, 48, 16, 3), (112, 96, 16, 13), (330, 1020, 10, 10),
    (1120, 1100, 20, 9), (2056, 1608, 8, 9),
])
@pytest.mark.parametrize("op,dtype", [("heat", "f64"), ("heat_kahan", "f32"), ("heat_kahan", "bf16")])
def test_march_edges_match_the_oracle(oracle_lib, op, dtype, nx, ny, tile, nsteps):
    u = 1.0 + np.random.default_rng(nx).random((ny, nx))
    if op == "heat":
        ref = oracle_lib.heat(u, 0.2, nsteps)
        assert np.array_equal(swept(op, u, nsteps, tile, (0.2,))[0], ref)
        return
    u = u.astype(np.float32)
    if dtype == "bf16":
        u = torch.from_numpy(u).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    ref_u, ref_c = oracle_lib.heat_kahan(u, np.zeros_like(u), 0.2, nsteps, storage=dtype)
    got = swept(op, np.stack([u, np.zeros_like(u)]), nsteps, tile, (0.2,), dtype=dtype)
    assert np.array_equal(got[0], ref_u) and np.array_equal(got[1], ref_c)


def test_batch_of_odd_and_even_grids_matches_the_oracle(oracle_lib):
    """Odd sides put the grids after them at odd offsets of the pool, where a
    pair of columns is not an aligned pair."""
    sizes = [(33, 47, 0), (64, 96, 32), (35, 31, 0), (130, 60, 10), (7, 5, 0)]
    us = [1.0 + np.random.default_rng(i).random((ny, nx)) for i, (nx, ny, _) in enumerate(sizes)]
    with SweptBatch([s[0] for s in sizes], [s[1] for s in sizes], [s[2] for s in sizes],
                    op="heat", params=(0.2,)) as b:
        b.set_state([u[None] for u in us])
        b.advance(23)
        got = b.split(b.get_state())
    for u, g in zip(us, got):
        assert np.array_equal(g[0], oracle_lib.heat(u, 0.2, 23))


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 1022, 2.0 ** 1023 * 1.2, 2.0 ** -1074 * 9])
def test_wave_fused_difference_has_the_bits_of_two_operations(oracle_lib, scale):
    """2u - u_old as one operation, also where 2u overflows, at infinities and
    zeros of both signs and below the normal numbers."""
    rng = np.random.default_rng(3)
    u = (1.0 + 0.4 * rng.random((2, 48, 64))) * scale
    u[0, 3, 4], u[1, 9, 9], u[0, 20:24, 20:24], u[1, 20:22] = np.inf, -np.inf, -0.0, 0.0
    with np.errstate(all="ignore"):
        ref_u, ref_old = oracle_lib.wave(u[0], u[1], 0.3 * 0.3, 11)
    got = swept("wave", u, 11, 16, (0.3,))
    assert np.array_equal(got[0], ref_u, equal_nan=True)
    assert np.array_equal(got[1], ref_old, equal_nan=True)


@pytest.mark.parametrize("mode", ["swept", "naive"])
def test_wave_difference_where_the_double_overflows(mode):
    """u of both signs in the last binade, whose double is an infinity, over old
    values that are NaN, infinities of either sign, and finite: one step against
    the update's operations one by one. (4u overflows there, too: the fused d is
    the neighbours' sum where that is an infinity, and -4u's infinity elsewhere.)"""
    u, old = np.full((16, 32), 1e308), np.zeros((16, 32))
    u[:, 16:] = -1.5e308
    old[:] = np.tile([np.nan, np.inf, -np.inf, 1e308, -1e308, 0.0, -0.0, 3.0], (16, 4))
    with np.errstate(all="ignore"):
        s = (np.roll(u, -1, 1) + np.roll(u, -1, 0)) + (np.roll(u, 1, 1) + np.roll(u, 1, 0))
        d = np.where(np.isinf(s), s, s - 4.0 * u)
        want = 0.3 * 0.3 * d + (2.0 * u - old)
    assert np.isnan(want).any() and np.isinf(want).any()
    with Swept2D(32, 16, op="wave", tile=4, params=(0.3,)) as sw:
        sw.set_state(np.stack([u, old]))
        sw.advance(1, mode=mode)
        got = sw.get_state()
    assert np.array_equal(got[0], want, equal_nan=True)
    assert np.array_equal(got[1], u)


@pytest.mark.parametrize("nx,ny,tile", [(64, 64, 16), (4, 4, 4), (768, 768, 16)])
def test_static_advance_makes_a_timed_out_wait_visible(oracle_lib, nx, ny, tile):
    """The call without a handle: u_out is NaN everywhere after a wait that gave
    up, and the next call is not touched by it."""
    import ctypes
    from paper_1602_07558_gb300.swept2d import EINVAL, OK, heat_advance_static, lib
    u0 = inputs.uniform(nx, ny, seed=4)
    d_in = torch.from_numpy(u0).to("cuda")
    d_out = torch.zeros_like(d_in)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    f = lib().swept2d_selftest_static_timeout
    f.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] * 3 + [ctypes.c_double, ctypes.c_longlong] \
        + [ctypes.c_void_p, ctypes.c_char_p, ctypes.c_int]
    call = lambda limit: f(d_in.data_ptr(), d_out.data_ptr(), nx, ny, tile, 0.2, limit,
                           stream.cuda_stream, None, 0)
    assert call(0) == EINVAL
    assert call(1000) == OK
    stream.synchronize()
    assert torch.isnan(d_out).all()
    assert np.array_equal(d_in.cpu().numpy(), u0)
    heat_advance_static(d_in, d_out, nx, ny, tile, 0.2, 13, stream=stream)
    stream.synchronize()
    assert np.array_equal(d_out.cpu().numpy(), oracle_lib.heat(u0, 0.2, 13))


@pytest.mark.parametrize("nx,ny,tile,nsteps", [
    (4, 4, 4, 3), (16, 60, 4, 4), (30, 30, 6, 5), (64, 48, 16, 6), (150, 150, 10, 3),
    (330, 300, 10, 3), (1040, 1056, 16, 2),
])
@pytest.mark.parametrize("op,dtype", [("euler_rk2", "f64"), ("euler_kahan", "f32"),
                                      ("euler_kahan", "bf16")])
def test_euler_march_edges_match_the_oracle(oracle_lib, op, dtype, nx, ny, tile, nsteps):
    """Each shape of the marching form and, in binary64, the sizes that stay with
    the swept kernels; every plane (binary64: U) bit for bit."""
    U = inputs.euler_pulse(nx, ny, 4, gamma=1.4)
    if op == "euler_rk2":
        u0 = np.concatenate([U, U])
        a, dt = oracle_lib.euler_setup(U, 1.4, 0.3)
        ref = oracle_lib.euler_rk2(U, 1.4, dt, 0.5, a, nsteps)
    else:
        U = U.astype(np.float32)
        if dtype == "bf16":
            U = torch.from_numpy(U).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
        Uf = (oracle_lib.bf16_bits_to_f32(U) if dtype == "bf16" else U).astype(np.float64)
        u0 = np.concatenate([U, U, np.zeros_like(U)])
        a, dt = oracle_lib.euler_setup(Uf, 1.4, 0.3)
        ref = oracle_lib.euler_kahan(u0, 1.4, dt, 0.5, a, nsteps, dtype)
    got = swept(op, u0, nsteps, tile, (1.4, 0.3, 0.5), dtype=dtype)
    assert np.array_equal(got[:len(ref)], ref)
    with Swept2D(nx, ny, op=op, tile=tile, params=(1.4, 0.3, 0.5), dtype=dtype) as s:
        s.set_state(u0)
        s.advance(nsteps, mode="naive")
        assert np.array_equal(got, s.get_state())      # the midpoint planes, too


def test_euler_batch_of_uneven_grids_matches_the_single_grids():
    sizes = [(33, 47, 0), (64, 96, 32), (35, 31, 0), (130, 60, 10)]
    for op, dtype in (("euler_rk2", "f64"), ("euler_kahan", "f32")):
        states = []
        for i, (nx, ny, _) in enumerate(sizes):
            U = inputs.euler_pulse(nx, ny, i, gamma=1.4)
            states.append(np.concatenate([U, U] + ([np.zeros_like(U)] if dtype == "f32" else []))
                          .astype(np.float32 if dtype == "f32" else np.float64))
        with SweptBatch([s[0] for s in sizes], [s[1] for s in sizes], [s[2] for s in sizes], op=op,
                        params=(1.4, 0.3, 0.5), dtype=dtype) as b:
            b.set_state(states)
            b.advance(7)
            got = b.split(b.get_state())
        for (nx, ny, _), u, g in zip(sizes, states, got):
            with Swept2D(nx, ny, op=op, tile=0, params=(1.4, 0.3, 0.5), dtype=dtype) as s:
                s.set_state(u)
                s.advance(7, mode="naive")
                assert np.array_equal(g, s.get_state())


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (29, 31), (30, 33), (31, 8), (61, 700), (1009, 757)])
@pytest.mark.parametrize("kind", ["one_binade", "crossing", "noise"])
def test_naive_heat_rows_and_launches_match_the_oracle(oracle_lib, kind, nx, ny):
    """The naive kernel's column chunks and rows a warp (one, FP64 only, to
    eight), in launches that follow each other without a gap, also in a graph."""
    u0 = field(kind, nx, ny) if kind == "noise" or min(nx, ny) > 2 else np.full((ny, nx), 1.25)
    ref = oracle_lib.heat(u0, 0.2, 13)
    with Swept2D(nx, ny, op="heat", tile=0, params=(0.2,), stream=torch.cuda.Stream()) as s:
        for graph in (False, True):
            s.set_state(u0[None])
            s.advance(13, mode="naive", graph=graph)
            assert np.array_equal(s.get_state()[0], ref)


@pytest.mark.parametrize("nx,ny", [(1, 65535 * 64 + 3), (2, 65535 * 64)])
def test_naive_heat_takes_more_rows_than_a_launch_has_blocks_along_y(oracle_lib, nx, ny):
    u0 = np.random.default_rng(ny).random((ny, nx))
    with Swept2D(nx, ny, op="heat", tile=0, params=(0.2,)) as s:
        s.set_state(u0[None])
        s.advance(3, mode="naive")
        assert np.array_equal(s.get_state()[0], oracle_lib.heat(u0, 0.2, 3))


@pytest.mark.parametrize("op,dtype", [("euler_rk2", "f64"), ("euler_kahan", "f32"),
                                      ("euler_kahan", "bf16")])
@pytest.mark.parametrize("nx,ny", [(13, 7), (61, 62), (457, 449)])
def test_naive_euler_launches_match_the_oracle(oracle_lib, op, dtype, nx, ny):
    """The naive path's walks (binary64, and the larger binary32 / bfloat16
    grids), on odd sides that no tile divides, split over two advances."""
    U = inputs.euler_pulse(nx, ny, 4, gamma=1.4)
    if op == "euler_kahan":
        U = U.astype(np.float32)
        if dtype == "bf16":
            U = torch.from_numpy(U).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    Uf = (oracle_lib.bf16_bits_to_f32(U) if dtype == "bf16" else U).astype(np.float64)
    a, dt = oracle_lib.euler_setup(Uf, 1.4, 0.3)
    if op == "euler_rk2":
        u0, ref = np.concatenate([U, U]), oracle_lib.euler_rk2(U, 1.4, dt, 0.5, a, 5)
    else:
        u0 = np.concatenate([U, U, np.zeros_like(U)])
        ref = oracle_lib.euler_kahan(u0, 1.4, dt, 0.5, a, 5, dtype)
    with Swept2D(nx, ny, op=op, tile=0, params=(1.4, 0.3, 0.5), dtype=dtype,
                 stream=torch.cuda.Stream()) as s:
        s.set_state(u0)
        s.advance(2, mode="naive")
        s.advance(3, mode="naive", graph=True)
        got = s.get_state()
    assert np.array_equal(got[:len(ref)], ref)


@pytest.mark.parametrize("nx,ny", [(64, 512), (65, 1000), (1000, 65), (272, 1056), (512, 512),
                                   (1030, 1001)])
@pytest.mark.parametrize("op,dtype", [("euler_rk2", "f64"), ("euler_kahan", "f32"),
                                      ("euler_kahan", "bf16")])
def test_naive_euler_gives_the_same_bits_by_walks_and_by_points(oracle_lib, op, dtype, nx, ny):
    """Grids on both sides of the choice between a thread a point and the walks of
    each shape against the oracle; a batch of the one grid, which may choose the
    other, gives the same midpoint planes, too."""
    U = inputs.euler_pulse(nx, ny, 4, gamma=1.4)
    np_dtype = np.float64
    if op == "euler_kahan":
        U = U.astype(np.float32)
        np_dtype = np.float32
        if dtype == "bf16":
            U = torch.from_numpy(U).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
            np_dtype = np.uint16
    Uf = (oracle_lib.bf16_bits_to_f32(U) if dtype == "bf16" else U).astype(np.float64)
    a, dt = oracle_lib.euler_setup(Uf, 1.4, 0.3)
    u0 = np.concatenate([U, U] + ([np.zeros_like(U)] if op == "euler_kahan" else []))
    ref = oracle_lib.euler_rk2(U, 1.4, dt, 0.5, a, 3) if op == "euler_rk2" else \
        oracle_lib.euler_kahan(u0, 1.4, dt, 0.5, a, 3, dtype)
    with Swept2D(nx, ny, op=op, tile=0, params=(1.4, 0.3, 0.5), dtype=dtype) as s:
        s.set_state(u0)
        s.advance(1, mode="naive")
        s.advance(2, mode="naive")
        got = s.get_state()
    with SweptBatch([nx], [ny], [0], op=op, params=(1.4, 0.3, 0.5), dtype=dtype) as b:
        b.set_state([u0.astype(np_dtype)])
        b.advance(3, mode="naive")
        other = b.split(b.get_state())[0]
    assert np.array_equal(got[:len(ref)], ref)
    assert np.array_equal(got, other)


@pytest.mark.parametrize("mode,graph", [("swept", False), ("swept", True), ("persistent", False)])
@pytest.mark.parametrize("nx,ny,tile", [(64, 2048, 32), (384, 384, 32), (48, 512, 16), (128, 512, 32),
                                        (560, 70, 10), (2000, 40, 8)])
def test_binary64_euler_gives_the_same_bits_in_either_form(oracle_lib, nx, ny, tile, mode, graph):
    """Grids on both sides of the choice between the swept kernels and the marching
    form's shapes, which differs between the two swept modes; five steps (a tail of
    sub-steps that fill no half cycle), then three more."""
    U = inputs.euler_pulse(nx, ny, 4, gamma=1.4)
    a, dt = oracle_lib.euler_setup(U, 1.4, 0.3)
    ref = oracle_lib.euler_rk2(U, 1.4, dt, 0.5, a, 8)
    with Swept2D(nx, ny, op="euler_rk2", tile=tile, params=(1.4, 0.3, 0.5),
                 stream=torch.cuda.Stream()) as s:
        s.set_state(np.concatenate([U, U]))
        s.advance(5, mode=mode, graph=graph)
        s.advance(3, mode=mode, graph=graph)
        assert np.array_equal(s.get_state()[:4], ref)


@pytest.mark.parametrize("op,dtype,nx,ny,tile", [
    ("heat", "f64", 64, 48, 16), ("heat", "f64", 2048, 1024, 64), ("heat_kahan", "f32", 64, 48, 16),
    ("heat_kahan", "bf16", 64, 48, 16), ("euler_rk2", "f64", 80, 320, 40),
    ("euler_kahan", "f32", 64, 48, 16), ("euler_kahan", "bf16", 64, 48, 16),
    ("euler_kahan", "bf16", 64, 1664, 32)])
def test_short_advances_take_naive_launches_with_the_same_bits(op, dtype, nx, ny, tile):
    """Up to a few sub-steps an advance in a swept mode is one naive launch each; every
    split of eight steps, by stream and by graph, ends in the same state."""
    if op.startswith("euler"):
        U, params = inputs.euler_pulse(nx, ny, 4, gamma=1.4), (1.4, 0.3, 0.5)
        u0 = np.concatenate([U, U] + ([np.zeros_like(U)] if op == "euler_kahan" else []))
    else:
        u, params = 1.0 + np.random.default_rng(1).random((1, ny, nx)), (0.2,)
        u0 = np.concatenate([u] + ([np.zeros_like(u)] if op == "heat_kahan" else []))
    if dtype != "f64":
        u0 = u0.astype(np.float32)
    if dtype == "bf16":
        u0 = torch.from_numpy(u0).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    with Swept2D(nx, ny, op=op, tile=tile, params=params, dtype=dtype,
                 stream=torch.cuda.Stream()) as s:
        results = []
        for split in ([8], [1] * 8, [2] * 4, [3, 4, 1], [7, 1]):
            for mode, graph in (("swept", False), ("persistent", True), ("naive", False)):
                s.set_state(u0)
                launches = s.query("launches")
                for k in split:
                    s.advance(k, mode=mode, graph=graph)
                if split == [1] * 8:
                    assert s.query("launches") - launches == 8 * s.nstages
                results.append(s.get_state())
    assert all(np.array_equal(results[0], r) for r in results)


@pytest.mark.parametrize("r", [0.0625, 0.05, 0.01, 2.0 ** -11 * 1.3, 2.0 ** -11, 2.0 ** -11 * 0.99])
@pytest.mark.parametrize("kind", ["one_binade", "binades", "negative", "crossing", "noise",
                                  "mixed_sign_noise", "ties", "few_bits", "powers", "constant",
                                  "zeros", "tiny", "smallest_normal", "huge"])
def test_small_diffusion_numbers_are_bitwise_in_either_mode(oracle_lib, kind, r):
    u0 = field(kind, 96, 64)
    with np.errstate(all="ignore"):
        ref = oracle_lib.heat(u0, r, 21)
    with Swept2D(96, 64, op="heat", tile=32, params=(r,)) as s:
        for mode in ("swept", "naive"):
            s.set_state(u0[None])
            s.advance(21, mode=mode)
            assert np.array_equal(s.get_state()[0], ref, equal_nan=True)


@pytest.mark.parametrize("kind", ["signed", "crossing", "uniform", "half", "zeros", "nan"])
@pytest.mark.parametrize("nx,ny,tile,nsteps", [
    (1024, 512, 32, 7), (768, 768, 32, 8), (768, 768, 32, 9), (1010, 1010, 10, 10),
    (1022, 504, 14, 11), (712, 720, 8, 264), (1280, 400, 40, 264 + 13)])
def test_large_fp64_heat_grids_of_every_kind_of_field(oracle_lib, kind, nx, ny, tile, nsteps):
    """Grids whose form the field decides (integer units or the FP64 walks): step
    counts of either parity, with a phase that only copies, and over two decisions;
    in the modes, as a graph, and by the call without a handle."""
    from paper_1602_07558_gb300.swept2d import SweptError, heat_advance_static
    rng = np.random.default_rng(nx)
    u0 = {"signed": lambda: 2 * rng.random((ny, nx)) - 1, "zeros": lambda: np.zeros((ny, nx)),
          "crossing": lambda: inputs.smooth_field(nx, ny, seed=2),
          "half": lambda: 1.5 + rng.random((ny, nx)), "uniform": lambda: rng.random((ny, nx)),
          "nan": lambda: 1.0 + rng.random((ny, nx))}[kind]()
    if kind == "half":
        u0[:, :nx // 2] -= 2.0
    if kind == "nan":
        u0[5, 6], u0[300, 400] = np.nan, np.inf
    with np.errstate(all="ignore"):
        ref = oracle_lib.heat(u0, 0.2, nsteps)
    with Swept2D(nx, ny, op="heat", tile=tile, params=(0.2,), stream=torch.cuda.Stream()) as s:
        for mode, graph in (("swept", False), ("swept", True), ("persistent", False)):
            s.set_state(u0[None])
            s.advance(nsteps, mode=mode, graph=graph)
            assert np.array_equal(s.get_state()[0], ref, equal_nan=True)
    d_in = torch.from_numpy(u0).to("cuda")
    d_out = torch.zeros_like(d_in)
    stream = torch.cuda.current_stream()
    try:
        heat_advance_static(d_in, d_out, nx, ny, 16 if nx % 16 == 0 and ny % 16 == 0 else tile,
                            0.2, nsteps, stream=stream)
    except SweptError as e:                     # (more panels than the scratch holds)
        assert "scratch" in str(e)
        return
    stream.synchronize()
    assert np.array_equal(d_out.cpu().numpy(), ref, equal_nan=True)


@pytest.mark.parametrize("r", [0.25, 0.3, -0.05, 2.0 ** -12])
@pytest.mark.parametrize("nx,ny,tile,nsteps", [
    (64, 48, 16, 21), (192, 384, 32, 37), (192, 384, 32, 16), (512, 512, 32, 34), (512, 512, 32, 33),
    (704, 720, 16, 19), (1000, 760, 40, 45)])
def test_diffusion_numbers_the_integer_units_cannot_take(oracle_lib, r, nx, ny, tile, nsteps):
    """The swept kernels (marching on small grids) and the naive walks, with tails of
    either parity, in every mode and by the call without a handle."""
    from paper_1602_07558_gb300.swept2d import heat_advance_static
    u0 = 2 * np.random.default_rng(nx).random((ny, nx)) - 1
    with np.errstate(all="ignore"):
        ref = oracle_lib.heat(u0, r, nsteps)
    with Swept2D(nx, ny, op="heat", tile=tile, params=(r,), stream=torch.cuda.Stream()) as s:
        for mode, graph in (("swept", False), ("swept", True), ("persistent", False),
                            ("naive", False), ("naive", True)):
            s.set_state(u0[None])
            s.advance(nsteps, mode=mode, graph=graph)
            assert np.array_equal(s.get_state()[0], ref)
    d_in = torch.from_numpy(u0).to("cuda")
    d_out = torch.zeros_like(d_in)
    heat_advance_static(d_in, d_out, nx, ny, tile, r, nsteps, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert np.array_equal(d_out.cpu().numpy(), ref) and np.array_equal(d_in.cpu().numpy(), u0)


@pytest.mark.parametrize("nx,ny,tile,nsteps", [(64, 2048, 32, 37), (64, 2048, 16, 20), (192, 384, 32, 53),
                                               (192, 384, 16, 25)])
@pytest.mark.parametrize("mode,graph", [("swept", False), ("swept", True), ("persistent", False)])
def test_fp64_heat_grids_that_keep_the_swept_kernels(oracle_lib, nx, ny, tile, nsteps, mode, graph):
    """Grids too narrow for the marching form's columns: the Up, Bridge, Octahedron and
    Down launches without a gap between them, with odd tails, twice in a row."""
    u0 = inputs.smooth_field(nx, ny, seed=3)
    ref = oracle_lib.heat(u0, 0.2, 2 * nsteps)
    with Swept2D(nx, ny, op="heat", tile=tile, params=(0.2,), stream=torch.cuda.Stream()) as s:
        s.set_timing(not graph)
        s.set_state(u0[None])
        s.advance(nsteps, mode=mode, graph=graph)
        s.advance(nsteps, mode=mode, graph=graph)
        assert np.array_equal(s.get_state()[0], ref)
        if not graph:
            assert s.kernel_stats("octahedron")[0] > 0 and s.kernel_stats("march")[0] == 0


@pytest.mark.parametrize("threads,stage", [(256, False), (128, True)])
@pytest.mark.parametrize("op,dtype,tile", [("heat_kahan", "f32", 16), ("heat_kahan", "bf16", 32),
                                           ("euler_kahan", "f32", 16), ("euler_kahan", "bf16", 8)])
def test_traced_persistent_advance_of_the_updates_that_march(oracle_lib, op, dtype, tile, threads, stage):
    """A trace records the persistent swept kernel's items, which nothing else runs for
    these updates: same bits as the marching advance, every item timed."""
    nx, ny, steps = 96, 64, 21
    if op == "heat_kahan":
        u, params, nst = 1.0 + np.random.default_rng(2).random((1, ny, nx)), (0.2,), 1
        u0 = np.concatenate([u, np.zeros_like(u)]).astype(np.float32)
    else:
        U, params, nst = inputs.euler_pulse(nx, ny, 4, gamma=1.4), (1.4, 0.3, 0.5), 2
        u0 = np.concatenate([U, U, np.zeros_like(U)]).astype(np.float32)
    if dtype == "bf16":
        u0 = torch.from_numpy(u0).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    tiles, halves = (nx // tile) * (ny // tile), steps * nst // (tile // 2)
    buf = torch.zeros(2 * tiles * (1 + 3 * halves), dtype=torch.int32, device="cuda")
    with Swept2D(nx, ny, op=op, tile=tile, params=params, dtype=dtype,
                 stream=torch.cuda.Stream()) as s:
        s.set_state(u0)
        s.advance(steps, mode="persistent")
        want = s.get_state()
        s.set_tuning(threads, stage)
        s.set_trace(buf)
        for graph in (False, True):
            s.set_state(u0)
            s.advance(steps, mode="persistent", graph=graph)
            assert np.array_equal(s.get_state(), want)
    assert (buf.cpu().numpy().view(np.uint32).reshape(-1, 2)[:, 1] > 0).all()


@pytest.mark.parametrize("op,dtype,params,march", [
    ("heat", "f64", (0.2,), True), ("heat", "f64", (0.25,), False), ("heat_kahan", "bf16", (0.2,), True),
    ("wave", "f64", (0.3,), False)])
def test_autotune_times_one_launch_shape_of_a_form_that_ignores_it(op, dtype, params, march):
    from paper_1602_07558_gb300.autotune import autotune, autotune_batch
    (tile, threads, _), table = autotune(256, 256, op, params, dtype=dtype, tiles=(16, 32), threads=(128, 256))
    rows = [r for r in table if "tile" in r]
    assert all(r["march"] == march for r in rows)
    assert len(rows) == 2 if march else len(rows) > 2
    assert (tile, threads) == (32, 256) if march else tile in (16, 32)
    if op != "wave":
        tiles, tuning, table = autotune_batch([64] * 3, [64] * 3, op, params, dtype=dtype, tiles=(16, 32),
                                              threads=(128, 256), probe_steps=16,
                                              stream=torch.cuda.Stream())
        assert [r["march"] for r in table if "tile" in r] == [True, True]   # (12,288 points)
        assert tiles == [32] * 3 and list(tuning) == [32]


@pytest.mark.parametrize("nx,ny", [(1, 500_001), (2, 300_001), (3, 200_001), (61, 9_001), (62, 9_000),
                                   (63, 8_999), (125, 4_001), (9_001, 61)])
def test_fp64_walks_on_narrow_and_odd_grids(oracle_lib, nx, ny):
    """The naive walks of an r off the integer units: fewer columns than lanes, tiles
    of the most and the fewest columns, odd sides."""
    u0 = 2 * np.random.default_rng(nx).random((ny, nx)) - 1
    with Swept2D(nx, ny, op="heat", tile=0, params=(0.25,), stream=torch.cuda.Stream()) as s:
        for graph in (False, True):
            s.set_state(u0[None])
            s.advance(5, mode="naive", graph=graph)
            assert np.array_equal(s.get_state()[0], oracle_lib.heat(u0, 0.25, 5))


@pytest.mark.parametrize("kind", ["signed", "uniform", "one_sign"])
@pytest.mark.parametrize("nx,ny,tile,nsteps", [(8, 65_536, 8, 8), (65_536, 8, 8, 13), (56, 9_184, 8, 9)])
def test_static_advance_of_large_narrow_grids(oracle_lib, kind, nx, ny, tile, nsteps):
    """Whose form the field decides, with fewer columns or rows than a tile has."""
    from paper_1602_07558_gb300.swept2d import heat_advance_static
    u0 = np.random.default_rng(ny).random((ny, nx))
    u0 = {"signed": 2 * u0 - 1, "uniform": u0, "one_sign": -1 - u0}[kind]
    d_in = torch.from_numpy(u0).to("cuda")
    d_out = torch.zeros_like(d_in)
    heat_advance_static(d_in, d_out, nx, ny, tile, 0.2, nsteps, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert np.array_equal(d_out.cpu().numpy(), oracle_lib.heat(u0, 0.2, nsteps))
