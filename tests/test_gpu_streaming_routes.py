"""The step's tests once more on the streaming kernels: a call of at most
400,000 cells without a launch shape runs one cell per lane in a single
kernel, so here the same cells are stepped under an explicit shape, which
reaches the ring, its cold chunks, the tails, the records and the queue at
every size: one and two cells per lane (the lean kernel wherever the arrays
allow it) and four (the general one)."""
import ctypes
import itertools

import pytest
import torch

import test_gpu_field as F
import test_gpu_multistep as M
import test_gpu_orbital as O
import test_gpu_small_grids as G
import test_gpu_step as S
import test_gpu_window_policy as P
from paper_2202_10647_gb300 import ionize, workloads as W

pytestmark = pytest.mark.gpu

# tests, and whether a single species under the paper's window rule lies in
# aligned arrays there (the lean kernel's)
TESTS = [(S.test_nitrogen_grid_parity, True), (S.test_fp32_coefficient_modes, True),
         (S.test_ladder_parity, True), (S.test_adversarial_cells, False),
         (S.test_time_steps_and_gas_density, True),
         (S.test_invalid_windows_are_skipped_and_counted, True),
         (S.test_cell_ranges_with_offset, False),
         (S.test_cold_chunks, False), (S.test_stiff_windows_rate_order, False),
         (S.test_near_degenerate_pairs_take_fp64_coefficients, False),
         (S.test_close_ends_far_inner_node, False),
         (S.test_fp64_coefficients_for_many_cells, True),
         (S.test_smallest_and_largest_species, False),
         (S.test_batched_smallest_with_largest_species, False),
         (O.test_step_with_l_and_m, False), (O.test_lognormal_cells_with_l_and_m, True),
         (F.test_step_field, False), (P.test_adaptive_policy_matches_oracle, False),
         (M.test_step_conservation_measure, False), (M.test_graph_with_fused_conservation, True)]


def cases():
    out = []
    for fn, lean in TESTS:
        marks = [m.args for m in getattr(fn, "pytestmark", []) if m.name == "parametrize"]
        axes = []
        for names, values in marks:
            names = [s.strip() for s in names.split(",")]
            axes.append([dict(zip(names, v if len(names) > 1 else (v,))) for v in values])
        for combo in itertools.product(*axes):
            kw = {k: v for d in combo for k, v in d.items()}
            if kw.get("flags", 0) & ionize.ION_F64_PLAIN or "FP64" in str(kw.get("case")):
                continue  # the FP64 form has no such route
            name = "-".join([fn.__name__[5:], *map(str, kw.values())])
            out.append(pytest.param(fn, kw, lean, id=name))
    return out


class Streaming:
    """ionize.step, step_field and step_batched under a launch shape."""

    def __init__(self, shape):
        self.shape = ionize.LaunchShape(*shape)
        self.real, self.real_batched = ionize.step, ionize.step_batched
        self.lean = 0

    def saw(self, ws, n):
        # (smaller calls are a tail: all records)
        if n >= 32 * self.shape.cells_per_lane and not torch.cuda.is_current_stream_capturing():
            # header word 8, the next chunk to hand out: only the streaming kernels count it up
            assert int(ws[32:36].cpu().view(torch.int32)[0]) > 0

    def step(self, sp, E, N, k_lo, k_hi, dt, dne, n_gas=None, ws=None, eps_shift=1e-6,
             degen_gap=1e-3, flags=ionize.ION_F32, ncells=None, offset=0, window=None):
        if flags & ionize.ION_F64_PLAIN:
            return self.real(sp, E, N, k_lo, k_hi, dt, dne, n_gas=n_gas, ws=ws,
                             eps_shift=eps_shift, degen_gap=degen_gap, flags=flags,
                             ncells=ncells, offset=offset, window=window)
        n = E.numel() - offset if ncells is None else ncells
        if offset + n > min(t.numel() for t in (E, k_lo, k_hi, dne)):
            raise ValueError("offset/ncells outside the arrays")
        ws = ionize.workspace(n, flags, E.device) if ws is None else ws
        at = [ionize._ptr(t, offset) for t in (E, N, k_lo, k_hi, dne, n_gas)]
        Q, ld = self.shape.cells_per_lane, N.shape[1]
        self.lean += (window is None and Q < 4 and ld % Q == 0
                      and all(p % 16 == 0 for p in (at[0], at[2], at[3]))
                      and at[1] % (4 * Q) == 0 and at[4] % (4 * Q) == 0)
        job = (ionize._BatchJob * 1)(ionize._BatchJob(sp.handle.value, at[0], at[1], ld, n, at[2],
                                                      at[3], at[4], at[5]))
        opts = ionize._opts(eps_shift, degen_gap, window)
        ionize._check(ionize.lib().ion_step_batched(
            job, 1, float(dt), ctypes.byref(opts), int(flags), ctypes.byref(self.shape),
            ionize._ptr(ws), ws.numel(), ionize._stream(E)))
        self.saw(ws, n)
        return ws

    def step_field(self, sp, components, N, k_lo, k_hi, dt, dne, ws=None, **kw):
        E = ionize.field_magnitude(*components)
        return self.step(sp, E, N, k_lo, k_hi, dt, dne, **kw)

    def step_batched(self, jobs, dt, **kw):
        ws = self.real_batched(jobs, dt, **dict(kw, shape=kw.get("shape") or self.shape))
        self.saw(ws, max(j[1].numel() for j in jobs))
        return ws


@pytest.mark.parametrize("shape", [(2, 8, 0), (1, 8, 0), (4, 4, 0)], ids=str)
@pytest.mark.parametrize("fn,kw,lean", cases())
def test_under_a_shape(fn, kw, lean, shape, monkeypatch):
    s = Streaming(shape)
    for name in ("step", "step_field", "step_batched"):
        monkeypatch.setattr(ionize, name, getattr(s, name))
    if fn is S.test_cold_chunks and shape[0] == 4:
        pytest.skip("its cold chunks are 64 cells long")
    fn(**kw)
    assert s.lean or not lean or shape[0] == 4


@pytest.mark.parametrize("name", ["N", "Kr-like"])
@pytest.mark.parametrize("flags", [0, ionize.ION_NO_WINDOW_UPDATE, ionize.ION_CONSERVATION_CHECK,
                                   ionize.ION_FORCE_FP64_COEF])
@pytest.mark.parametrize("n", [61, 125, 20_009])
def test_direct_and_lean_grids(name, flags, n):
    """Single states, invalid windows, zero and negative fields, a gas density and the step's own
    conservation measure on the lean kernel: rows of a multiple of four cells."""
    assert (n + 3) % 4 == 0
    G.test_direct_and_streaming_grids(name, flags, None, n)


@pytest.mark.parametrize("shape", [(2, 8, 0), (1, 8, 0), (4, 4, 0)], ids=str)
@pytest.mark.parametrize("guard", [16, 12])
def test_guard_cells_untouched(guard, shape):
    """Canaries: planes and cells around the arrays stay bit-identical (16 cells in, the lean
    kernel; 12, windows that are not 16-byte aligned)."""
    wl = W.nitrogen_3d(8, 16, 32, seed=14)
    n, Z = wl.ncells, 7
    s = Streaming(shape)
    big = torch.full((Z + 3, n + 2 * guard), 12345.0, device="cuda")
    big[1:Z + 2, guard:guard + n] = wl.N[:, :n].cuda()

    def framed(t, value):
        b = torch.full((n + 2 * guard,), value, dtype=t.dtype, device="cuda")
        b[guard:guard + n] = t.cuda()
        return b

    E, lo, hi = framed(wl.E, 777.0), framed(wl.lo, 200), framed(wl.hi, 200)
    dne = framed(torch.zeros(n), 5.5)
    s.step(S.gpu_species(wl.species), E, big[1:Z + 2], lo, hi, 0.05, dne, offset=guard, ncells=n)
    assert s.lean == (guard == 16 and shape[0] < 4)
    b = big.cpu()
    assert torch.all(b[0] == 12345.0) and torch.all(b[Z + 2] == 12345.0)
    assert not torch.equal(b[1:Z + 2, guard:guard + n], wl.N[:, :n])
    for t, v in ((b[1:Z + 2].T, 12345.0), (dne, 5.5), (lo, 200), (hi, 200)):
        assert torch.all(t[:guard] == v) and torch.all(t[guard + n:] == v)
