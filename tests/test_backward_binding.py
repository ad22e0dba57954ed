"""What the binding of the two backward calls passes on to the library and what it refuses itself, on the CPU:
tensors that say they are on a GPU, and a library that writes down its calls."""
import pytest
import torch

from paper_2603_02561_b200 import solar

B, N, M, d, r = 2, 10, 5, 32, 3


class Gpu:
    def __init__(self, t, cuda=True):
        self.t, self.dtype, self.shape, self.device, self.is_cuda = t, t.dtype, t.shape, t.device, cuda

    def numel(self): return self.t.numel()
    def is_contiguous(self): return self.t.is_contiguous()
    def data_ptr(self): return self.t.data_ptr()


class Recorder:
    def __init__(self): self.calls = []

    def __getattr__(self, name):
        if not name.startswith("solar_"):
            raise AttributeError(name)
        if name == "solar_status_string":
            return lambda st: b"status"
        return lambda *a: (self.calls.append((name, a)), 0)[1]


@pytest.fixture
def library(monkeypatch):
    rec = Recorder()
    monkeypatch.setattr(solar, "_lib", rec)
    monkeypatch.setattr(solar, "_stream", lambda stream=None: 0)
    return rec


def sizes(call, dt):
    if call == "attention":
        return {"C": ((B, M, d), dt), "S": ((B, r), torch.float32), "V": ((B, d, r), torch.float32),
                "Wq": ((d, d), dt), "Wk": ((d, d), dt), "Wv": ((d, d), dt), "dO": ((B, M, d), dt)}
    return {"H": ((B, N, d), dt), "S": ((B, r), torch.float32), "V": ((B, d, r), torch.float32),
            "dS": ((B, r), torch.float32), "dV": ((B, d, r), torch.float32), "dH": ((B, N, d), dt)}


def run(call, t):
    ws = Gpu(torch.empty(1 << 20, dtype=torch.uint8))
    if call == "attention":
        solar.svd_attention_bwd(t["C"], t["S"], t["V"], t["Wq"], t["Wk"], t["Wv"], 0.1, t["dO"], ws)
    else:
        solar.svd_backward(t["H"], t["S"], t["V"], t["dS"], t["dV"], t["dH"], ws)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("call", ["attention", "svd"])
def test_backward_calls_look_at_every_tensor(library, call, dt):
    want = sizes(call, dt)
    good = {k: Gpu(torch.zeros(s, dtype=t)) for k, (s, t) in want.items()}
    run(call, good)
    assert len(library.calls) == 1
    first = {"attention": "C", "svd": "H"}[call]                 # its type is the call's storage type
    for name, (shape, t) in want.items():
        wrong = [Gpu(torch.zeros(shape, dtype=t), cuda=False), Gpu(torch.zeros((*shape[:-1], 2 * shape[-1]), dtype=t)[..., ::2])]
        if name != first:
            wrong.append(Gpu(torch.zeros(shape, dtype=torch.bfloat16 if t is torch.float32 else torch.float32)))
        if name not in (first, "V", "S") or (name, call) == ("S", "svd"):      # (the sizes are read off these)
            wrong.append(Gpu(torch.zeros((shape[0] - 1, *shape[1:]), dtype=t)))
        for w in wrong:
            with pytest.raises(ValueError):
                run(call, {**good, name: w})
    assert len(library.calls) == 1


@pytest.mark.parametrize("call,names", [("attention", ("V", "Wq", "Wk", "Wv")), ("svd", ("S", "dS", "dV", "dH"))])
def test_missing_tensors_are_the_librarys_to_refuse(library, call, names):
    good = {k: Gpu(torch.zeros(s, dtype=t)) for k, (s, t) in sizes(call, torch.float32).items()}
    run(call, good)
    for name in names:
        run(call, {**good, name: None})
        assert library.calls[-1][1].count(None) == library.calls[0][1].count(None) + 1, name


def test_a_buffer_of_another_shape_is_taken(library):
    good = {k: Gpu(torch.zeros(s, dtype=t)) for k, (s, t) in sizes("svd", torch.float32).items()}
    run("svd", {**good, "dH": Gpu(torch.zeros(B * N + 1, d)), "dS": Gpu(torch.zeros(B * r, 1))})
    assert len(library.calls) == 1
