"""The starting shapes (each pass its own) survive tuning: they are part of the stored
state, come back when asked for, are tried by the autotuner, and a tuning that fails
leaves the shape that was there.  Shapes stored for another transform engine miss."""
import pytest

b = pytest.importorskip("paper_2606_06247_gb300.binding")


class StandIn(b.Context):
    def __init__(self):
        self.grid = b.fcsph_grid(256, 256, 1.0, 1.0, 1, 32, 1, 0.0)
        self.fc = b.fcsph_fc(b.FC_GRAM, 5, 25, 0)
        self.kernel = b.fcsph_kernel(b.FAMILY["G8"], 1.3)
        self.prec = b.fcsph_precision(b.PREC["f32x2"], 0)
        self.h = None
        self.calls = []
        for n in ("set_tiling", "set_cta_threads", "set_step_groups", "set_step_persistent", "set_auto_shape"):
            setattr(self, n, lambda *a, n=n: self.calls.append((n,) + a))

    def tune_state(self):
        return {"auto": True, "tiling": [1, 1], "cta_threads": [32, 64], "groups": 2, "persistent": False}

    def get_tiling(self):
        return 1, 1

    def _params(self, *a):
        return b.fcsph_step_params()


def test_stored_starting_shape_is_applied_as_such():
    ctx = StandIn()
    ctx.apply_tune_state(ctx.tune_state())
    assert ctx.calls == [("set_auto_shape", True), ("set_step_groups", 2), ("set_step_persistent", False)]
    ctx.calls.clear()
    ctx.apply_tune_state({"tiling": [2, 4], "cta_threads": [64, 128], "groups": 1, "persistent": True})
    assert ctx.calls == [("set_tiling", 2, 4), ("set_cta_threads", 64, 128), ("set_step_groups", 1),
                         ("set_step_persistent", True)]


def test_shape_of_another_engine_misses(tmp_path, monkeypatch):
    path = str(tmp_path / "tune.json")
    ctx = StandIn()
    key = ctx.tune_key("rk3", "GB300")
    b.store_tune_cache(path, key.split("|", 1)[1], ctx.tune_state())  # as the former engine's key named it
    calls = []
    monkeypatch.setattr(b.lib, "fcsph_autotune", lambda *a: calls.append(a) or 0, raising=False)
    ctx.autotune(steps=1, cache=path, device_name="GB300")
    assert len(calls) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32x2", "f32"])
def test_starting_shape_comes_back(prec):
    from gpu_common import binding, grid_lengths, torch_cuda
    torch = torch_cuda()
    binding()
    nx = ny = 40
    lx, ly = grid_lengths(nx, ny, True)
    ctx = b.Context(nx, ny, lx, ly, x_walls=True, batch=3, family="G8", prec=prec)
    f = torch.rand((3, nx, ny), device="cuda", dtype=torch.float32 if prec == "f32" else torch.float64)

    def run():
        o = [torch.zeros_like(f)]
        ctx.spectral_op(f, ["LAP"], o)
        ctx.sync()
        return o[0]
    start, ref = ctx.tune_state(), run()
    assert start["auto"]
    ctx.apply_tune_state(start)
    assert ctx.tune_state() == start
    ctx.set_tiling(2, 4)
    assert not ctx.get_auto_shape() and torch.equal(run(), ref)
    with pytest.raises(b.FcsphError):
        ctx.autotune(steps=1, dt=-1.0)
    assert not ctx.get_auto_shape() and ctx.get_tiling() == (2, 4)
    ctx.set_auto_shape(True)
    assert ctx.tune_state() == start and torch.equal(run(), ref)
    with pytest.raises(b.FcsphError):
        ctx.autotune(steps=1, dt=-1.0)
    assert ctx.tune_state() == start
    ctx.autotune(steps=1, nu=1e-3, dt=1e-5)
    tuned = ctx.tune_state()
    assert torch.equal(run(), ref)
    ctx.set_auto_shape(True)
    ctx.apply_tune_state(tuned)
    assert ctx.tune_state() == tuned and torch.equal(run(), ref)
