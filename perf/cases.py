"""The work that users of the Virtual-Expert MoE layer have it do, as measurable cases.

A case is a plain dict.  Its kinds are the ways a program drives the library:

``stack``  one step of a decode loop: a stack of layers behind ``DecodeStack.step_graph`` (one CUDA graph of all
           forwards, importance read every eight steps without a wait, resident sets that have converged)
``call``   one ``Layer.forward`` on the current stream; with ``scores`` the three per-expert scores are also copied out
           and zeroed (``read_scores_async``), which is how a prefill feeds the next choice of resident experts
``host``   one ``Layer.forward_host``: tokens in pinned host memory, result in pinned host memory
``swap``   two forwards while two experts trade places: each enters from pinned host memory through a spare arena
           entry on a side stream, and the slot table flips once its copy has landed

Sizes are those of the configurations in ``inputs.CONFIGS`` and of the tests' ranges (d_model and d_ff multiples of 64,
up to 256 experts, 64 slots and four experts per token), with ragged token counts between them.
"""
import numpy as np
import torch

from paper_2308_15030_b200 import binding
from paper_2308_15030_b200.decode import DecodeStack, LayerState

RUN_LEN = 32          # consecutive tokens of a sequence that share one preferred expert set
PREFERRED = 4         # its size
PULL_PROB = 0.9       # probability that a token is pulled towards its set ...
PULL = 12.0           # ... by this much on the logit of one member

# (d_model, d_ff): the configurations' layer shapes and widths around them, some no multiple of 128 or 256
RELU_SHAPES = [(768, 3072), (1024, 4096), (512, 2048), (704, 2240), (1536, 1088)]
GATED_SHAPES = [(4096, 14336), (1024, 3584), (2048, 5632), (960, 2624)]
FINE_SHAPES = [(1024, 512), (768, 768), (2048, 1024)]


def _case(kind, T, d, f, E, K, k=1, dtype="bf16", act="relu", renorm=False, zipf=0.0, layers=1, scores=False):
    return {"kind": kind, "T": T, "d": d, "f": f, "E": E, "K": K, "k": k, "dtype": dtype, "act": act,
            "renorm": renorm, "zipf": zipf, "layers": layers, "scores": scores}


def listed():
    return [
        # One user's decode step through twelve layers: the latency of a chain of single-token layers.
        dict(_case("stack", 1, 1024, 4096, 64, 16, zipf=1.1, layers=12), name="stack_1"),
        # The same with a few dozen concurrent streams: most slots touched by one or two tokens each.
        dict(_case("stack", 29, 1024, 4096, 64, 16, zipf=1.1, layers=12), name="stack_29"),
        # The smallest eager call: three tokens of one layer, launched by the program itself.
        dict(_case("call", 3, 768, 3072, 64, 16, zipf=1.1), name="call_3"),
        # A mid-size batch of a 64-expert encoder layer.
        dict(_case("call", 2048, 768, 3072, 64, 16, zipf=1.1), name="call_2048"),
        # Prefill of sixteen sequences of 512 tokens; the scores decide the next resident set.
        dict(_case("call", 8192, 768, 3072, 128, 32, zipf=1.0, scores=True), name="prefill_8192"),
        # Many small experts, four per token, every slot of the arena in use, ragged batch.
        dict(_case("call", 6011, 1024, 512, 256, 64, k=4, renorm=True, zipf=1.1), name="fine_6011"),
        # Wide gated experts: prefill (arithmetic-bound) and a small decode batch (weights-bound).
        dict(_case("call", 4096, 4096, 14336, 8, 4, k=2, act="swiglu", renorm=True), name="gated_4096"),
        dict(_case("call", 13, 4096, 14336, 8, 4, k=2, act="swiglu", renorm=True), name="gated_13"),
        # Single precision: the small ReLU layer, and a gated top-2 layer on a ragged batch.
        dict(_case("call", 256, 768, 3072, 8, 4, dtype="fp32"), name="fp32_256"),
        dict(_case("call", 1531, 1024, 2816, 16, 5, k=2, dtype="fp32", act="swiglu", renorm=True, zipf=1.1),
             name="fp32_gated_1531"),
        # A request served end to end from host memory, ragged length.
        dict(_case("host", 1999, 768, 3072, 64, 16, zipf=1.1), name="host_1999"),
        # Serving a full decode batch while experts are swapped over the host link.
        dict(_case("swap", 64, 1024, 4096, 64, 16, zipf=1.1), name="swap_64"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(lo * (hi / lo) ** rng.random() + rng.random()))


def draw(rng):
    kind = rng.choice(["stack", "call_relu", "call_relu", "call_relu", "call_gated", "call_gated", "call_fine",
                       "call_fp32", "call_fp32", "host", "swap"])
    zipf = rng.choice([0.0, 1.0, 1.1])
    if kind == "stack":
        d, f = rng.choice(RELU_SHAPES)
        return _case("stack", _log_int(rng, 1, 64), d, f, 64, rng.choice([8, 12, 16]), zipf=zipf,
                     layers=rng.randint(6, 12))
    if kind == "call_relu":
        d, f = rng.choice(RELU_SHAPES)
        E = rng.choice([8, 40, 64, 128, 256])
        return _case("call", _log_int(rng, 1, 16384), d, f, E, rng.randint(4, min(E, 48)), zipf=zipf,
                     scores=rng.random() < 0.3)
    if kind == "call_gated":
        d, f = rng.choice(GATED_SHAPES)
        E = rng.choice([8, 16])
        return _case("call", _log_int(rng, 1, 4000), d, f, E, 4, k=2, act="swiglu", renorm=True, zipf=zipf)
    if kind == "call_fine":
        d, f = rng.choice(FINE_SHAPES)
        return _case("call", _log_int(rng, 16, 8192), d, f, rng.choice([128, 256]), rng.randint(24, 64),
                     k=rng.randint(2, 4), act=rng.choice(["relu", "swiglu"]), renorm=True, zipf=zipf)
    if kind == "call_fp32":
        d, f = rng.choice(RELU_SHAPES)
        act = rng.choice(["relu", "swiglu"])
        k = 2 if act == "swiglu" else 1
        return _case("call", _log_int(rng, 1, 4096), d, f, rng.choice([8, 16, 64]), rng.randint(4, 8), k=k,
                     dtype="fp32", act=act, renorm=k > 1, zipf=zipf)
    d, f = rng.choice(RELU_SHAPES)
    if kind == "host":
        return _case("host", _log_int(rng, 16, 8192), d, f, 64, rng.randint(8, 32), zipf=zipf)
    return _case("swap", _log_int(rng, 1, 256), d, f, 64, rng.randint(8, 16), zipf=zipf)


# ------------------------------------------------------------------ inputs
def _dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _tokens(case, Wr, gen, run_len):
    """x ~ N(0,1); with ``zipf`` a token is pulled towards one expert of the set that its run of tokens prefers."""
    T, E = case["T"], case["E"]
    x = torch.randn(T, case["d"], device="cuda", generator=gen)
    if case["zipf"] > 0:
        law = torch.arange(1, E + 1, device="cuda", dtype=torch.float32) ** -case["zipf"]
        rank_to_id = torch.randperm(E, device="cuda", generator=gen)
        runs = -(-T // run_len)
        sets = torch.multinomial(law.expand(runs, E), min(PREFERRED, E), generator=gen)
        member = torch.randint(0, sets.shape[1], (T,), device="cuda", generator=gen)
        run = torch.arange(T, device="cuda") // run_len
        expert = rank_to_id[sets[run, member]]
        W = Wr.float()
        pull = PULL * W / (W * W).sum(1, keepdim=True)
        x += (torch.rand(T, 1, device="cuda", generator=gen) < PULL_PROB) * pull[expert]
    return x.to(_dtype(case))


def _weights(shape, dtype, gen):
    w = torch.empty(shape, dtype=dtype, device="cuda")
    return w.normal_(0.0, 0.02, generator=gen)


class _LayerInputs:
    """One layer with its weights in HBM and the most important experts of its tokens resident."""

    def __init__(self, case, gen, rng, run_len, spare=0):
        d, f, E, K = case["d"], case["f"], case["E"], case["K"]
        dt = _dtype(case)
        gated = case["act"] == "swiglu"
        self.Wr = torch.randn(E, d, device="cuda", generator=gen).mul_(0.1).to(dt)
        self.x = _tokens(case, self.Wr, gen, run_len)
        self.arena_in = _weights((K + spare, 2 if gated else 1, f, d), dt, gen)
        self.arena_out = _weights((K + spare, d, f), dt, gen)
        norm = 0.02 * float((3 if gated else 2) * d * f) ** 0.5
        self.enorm = (norm * (1.0 + 0.01 * rng.standard_normal(E))).astype(np.float32)
        self.layer = binding.Layer(E, d, f, case["k"], K, binding.F32 if case["dtype"] == "fp32" else binding.BF16,
                                   binding.ACT_SWIGLU if gated else binding.ACT_RELU, int(case["renorm"]),
                                   max_tokens=case["T"], spare_slots=spare)
        self.layer.set_router(self.Wr, self.enorm)
        self.layer.set_resident(np.arange(K, dtype=np.int32), self.arena_in, self.arena_out)
        self.out = torch.empty_like(self.x)
        self.layer.forward(self.x, self.out)
        order = binding.topk_importance(self.layer.read_importance(reset=True), E)
        for kind in ("count", "eq1_masked"):
            self.layer.read_score(kind, reset=True)
        self.s2e, self.rest = order[:K].copy(), order[K:]
        self.phys = np.arange(K, dtype=np.int32)
        self.layer.set_resident(self.s2e, self.arena_in, self.arena_out, self.phys)


class _State:
    pass


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    s = _State()
    s.kind, s.scores = case["kind"], None
    if case["kind"] == "stack":
        inputs = [_LayerInputs(case, gen, rng, 1) for _ in range(case["layers"])]
        s.x = torch.stack([i.x for i in inputs])
        # the sets have converged: no step of this loop loads an expert, so the host copies need no contents
        host = [torch.empty((1,) + tuple(a.shape[1:]), dtype=a.dtype).pin_memory().expand((case["E"],) + tuple(a.shape[1:]))
                for a in (inputs[0].arena_in, inputs[0].arena_out)]
        states = [LayerState(i.layer, i.s2e, i.phys, [], i.arena_in, i.arena_out, host[0], host[1], enorm=i.enorm)
                  for i in inputs]
        s.out = torch.empty_like(s.x)
        s.stack = DecodeStack(states, frequency=8, commit="ready", async_decide=True, max_in_flight=8,
                              graph_buffers=(torch.empty_like(s.x), s.out))
        return s
    s.inputs = i = _LayerInputs(case, gen, rng, 1 if case["kind"] == "swap" else RUN_LEN,
                                spare=1 if case["kind"] == "swap" else 0)
    if case["scores"]:
        s.scores = torch.zeros(3, case["E"], dtype=torch.float32).pin_memory()
    if case["kind"] == "host":
        s.x = i.x.cpu().pin_memory()
        s.out = torch.empty_like(s.x).pin_memory()
    elif case["kind"] == "swap":
        # slot 0 alternates between the most important expert and the best one that is not resident
        s.outs = [torch.empty_like(i.x), torch.empty_like(i.x)]
        s.experts = [int(i.rest[0]), int(i.s2e[0])]
        newcomer = [_weights(tuple(a.shape[1:]), a.dtype, gen) for a in (i.arena_in, i.arena_out)]
        s.host_in = [newcomer[0].cpu().pin_memory(), i.arena_in[0].cpu().pin_memory()]
        s.host_out = [newcomer[1].cpu().pin_memory(), i.arena_out[0].cpu().pin_memory()]
        s.entries = [case["K"], 0]
        s.side = torch.cuda.Stream()
        s.done = [torch.cuda.Event(), torch.cuda.Event()]
    return s


def run(s):
    if s.kind == "stack":
        s.stack.step_graph(s.x)
        return s.out
    i = s.inputs
    if s.kind == "host":
        i.layer.forward_host(s.x, s.out)
        return s.out
    if s.kind == "swap":
        compute = torch.cuda.current_stream()
        for n in (0, 1):
            i.layer.load_slot_async(s.entries[n], s.host_in[n], s.host_out[n], compute, s.side, s.done[n])
            i.layer.forward(i.x, s.outs[n])
            compute.wait_event(s.done[n])
            i.s2e[0], i.phys[0] = s.experts[n], s.entries[n]
            i.layer.set_resident(i.s2e, i.arena_in, i.arena_out, i.phys)
        return s.outs
    i.layer.forward(i.x, i.out)
    if s.scores is None:
        return i.out
    i.layer.read_scores_async(("eq1", "count", "eq1_masked"), s.scores, reset=True)
    return {"out": i.out, "scores": s.scores}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    nb = 4 if case["dtype"] == "fp32" else 2
    d, f, pairs = case["d"], case["f"], case["T"] * case["k"]
    matrices = 3 if case["act"] == "swiglu" else 2
    # slots that receive a token: the expected number if tokens choose among the resident experts alike
    touched = case["K"] * (1.0 - (1.0 - 1.0 / case["K"]) ** pairs)
    one_bytes = touched * matrices * d * f * nb + case["E"] * d * nb + 2 * case["T"] * d * nb
    one_flops = 2.0 * pairs * matrices * d * f + 2.0 * case["T"] * case["E"] * d
    forwards = 2 if case["kind"] == "swap" else case["layers"]
    return {"bytes": forwards * one_bytes, "flops": forwards * one_flops}


def tolerance(case):
    # Relative error (2-norm) against the same layer evaluated in 64 bits from the same routing, over forty cases: bf16
    # layers 2.3e-3 to 2.4e-3 (hidden activations and outputs are rounded to bf16); fp32 layers 7e-6 to 2.6e-5 (products
    # of two-piece operands, sums in the tensor core's accumulators).  About four times the largest.
    return {"rel": 1e-4} if case["dtype"] == "fp32" else {"rel": 1e-2}
