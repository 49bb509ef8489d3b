"""Performance cases of the framework: what a user of the Routing-Mamba layer library runs, through the public binding.

Entry points covered: the layer forward (training / prefill), its backward, the single-token step (generation), the FFN-MoE
that shares the layer's routing, and the layer on a Mamba2-style block.  Widths, expert counts and dtypes are those of the
seeded workloads in `paper_2506_18145_b200/synth.py`; the ragged cases change the token counts to ones that no tile divides.

Inputs are drawn on the GPU with O(1) activations at every stage (projection std 1/sqrt(fan_in)), so that every stage of the
layer, the recurrence included, shows in the result.  A is negative, near -(n+1) and not an arithmetic progression; the dt bias
gives steps log-uniform in [1e-3, 1e-1], as at the start of training.
"""
import math

import torch

from paper_2506_18145_b200 import binding as rb

N_STATE, D_CONV = 16, 4
HEADDIM = 64               # channels per head of the Mamba2-style block


def _case(name, op, B, L, d_model, E, K, dtype="bf16", skew=0.0):
    return {"name": name, "op": op, "B": B, "L": L, "d_model": d_model, "E": E, "K": K, "dtype": dtype, "skew": skew}


def listed():
    return [
        # interactive generation: one sequence, one token per call; latency and launches
        _case("decode_1", "step", 1, 1, 2048, 8, 1),
        # a serving batch that generates in lock-step (the batch of the benchmark's step stage)
        _case("decode_64", "step", 64, 1, 2048, 8, 1),
        # the fp32 configuration: a small model checked or debugged in full precision
        _case("forward_tiny_fp32", "forward", 1, 256, 256, 4, 1, "f32"),
        # one layer of the 353M model on a small training batch
        _case("forward_small", "forward", 4, 2048, 1024, 8, 1),
        # prefill of a few prompts of an awkward length, two experts per token
        _case("forward_ragged", "forward", 3, 1017, 1536, 8, 2),
        # the headline benchmark: one 16384-token sequence through a 1.3B layer
        _case("forward_long", "forward", 1, 16384, 2048, 8, 1),
        # a training batch with sixteen experts, two per token, and a skewed router (busiest expert about 5x the mean)
        _case("forward_zipf", "forward", 8, 4096, 2048, 16, 2, skew=0.657),
        # a large training batch of short sequences: the largest forward
        _case("forward_short_seqs", "forward", 64, 1024, 1536, 8, 2),
        # training: backward of a small top-2 layer, lengths that no tile divides
        _case("backward_ragged", "backward", 3, 1371, 1024, 8, 2),
        # training: backward at the headline shape
        _case("backward_long", "backward", 1, 16384, 2048, 8, 1),
        # the hybrid model's FFN-MoE behind a layer of the headline shape, hidden width 4 x d_model
        _case("ffn_long", "ffn", 1, 16384, 2048, 8, 1),
        # routing on a Mamba2-style block at the headline shape
        _case("mamba2_long", "mamba2", 1, 16384, 2048, 8, 1),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    op = rng.choice(["step", "step", "forward", "forward", "forward", "forward", "backward", "backward", "ffn", "mamba2"])
    E, K = rng.choice([4, 8, 8, 16]), rng.choice([1, 1, 2])
    skew = rng.choice([0.0, 0.0, 0.657])
    if op == "step":
        return _pure(_case("", op, _log_int(rng, 1, 256), 1, 256 * rng.randint(4, 8), E, K))
    if op == "forward" and rng.random() < 0.2:      # the fp32 configuration stays small
        return _pure(_case("", op, rng.randint(1, 2), _log_int(rng, 64, 2048), 64 * rng.randint(2, 8), 4, K, "f32"))
    d_model = 512 * rng.randint(2, 4) if op == "mamba2" else 64 * rng.randint(12, 32)
    tokens = _log_int(rng, 700, (24576 if K == 1 else 12288) if op in ("forward", "ffn", "mamba2") else (12288 if K == 1 else 6144))
    B = min(tokens // 64, _log_int(rng, 1, 48))
    return _pure(_case("", op, B, tokens // B, d_model, E, K, skew=skew))


def _pure(c):
    del c["name"]
    return c


def _dims(c):
    d_model = c["d_model"]
    return d_model, 2 * d_model, -(-(d_model // 16) // 16) * 16        # D_m, D_e, dt rank (a multiple of 16)


class _Draw:
    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.dtype = torch.float32 if dtype == "f32" else torch.bfloat16

    def normal(self, shape, std=1.0, dtype=None):
        return torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32).mul_(std).to(dtype or self.dtype)

    def normal32(self, shape, std=1.0):
        return self.normal(shape, std, torch.float32)

    def uniform(self, shape):
        return torch.rand(shape, generator=self.g, device="cuda", dtype=torch.float32)

    def dt_bias(self, n):
        dt0 = torch.exp(self.uniform((n,)) * (math.log(1e-1) - math.log(1e-3)) + math.log(1e-3))
        return dt0 + torch.log(-torch.expm1(-dt0))


def _router(d, c, d_model):
    W_r = d.normal((c["E"], d_model), 0.9 / math.sqrt(d_model))
    b_r = -c["skew"] * 1.2 * torch.log(torch.arange(1, c["E"] + 1, dtype=torch.float32, device="cuda")) if c["skew"] else None
    return W_r, b_r


def _layer_weights(d, c):
    Dm, De, R = _dims(c)
    E = c["E"]
    W_r, b_r = _router(d, c, Dm)
    n = torch.arange(1, N_STATE + 1, dtype=torch.float32, device="cuda")
    return {"W_r": W_r, "b_r": b_r, "W_inz": d.normal((E, 2 * De, Dm), Dm ** -0.5), "w_conv": d.normal((D_CONV, De), 0.5),
            "b_conv": d.normal32((De,), 0.1), "W_x": d.normal((R + 2 * N_STATE, De), De ** -0.5), "W_dt": d.normal((De, R), R ** -0.5),
            "b_dt": d.dt_bias(De), "A": (-n[None, :] * (0.5 + d.uniform((De, N_STATE)))).contiguous(),
            "D": 1.0 + d.normal32((De,), 0.1), "W_out": d.normal((E, Dm, De), De ** -0.5)}


def _mamba2_weights(d, c):
    Dm, De, _ = _dims(c)
    E, H = c["E"], De // HEADDIM
    W_r, b_r = _router(d, c, Dm)
    return {"W_r": W_r, "b_r": b_r, "W_in": d.normal((E, 2 * De + 2 * N_STATE + H, Dm), Dm ** -0.5),
            "w_conv": d.normal((D_CONV, De + 2 * N_STATE), 0.5), "b_conv": d.normal32((De + 2 * N_STATE,), 0.1), "dt_bias": d.dt_bias(H),
            "A": -(0.5 + d.uniform((H,))) * (1.0 + torch.arange(H, device="cuda", dtype=torch.float32) % 8), "D": 1.0 + d.normal32((H,), 0.1),
            "w_norm": 1.0 + d.normal32((De,), 0.1), "W_out": d.normal((E, Dm, De), De ** -0.5)}


def prepare(case, seed):
    c, op = case, case["op"]
    d = _Draw(seed, c["dtype"])
    Dm, De, R = _dims(c)
    B, L, E, K = c["B"], c["L"], c["E"], c["K"]
    T = B * L
    empty = lambda shape, dtype: torch.empty(shape, dtype=dtype, device="cuda")  # noqa: E731
    cfg = rb.make_config(B, L, Dm, De, N_STATE, D_CONV, R, E, K, c["dtype"])
    x = d.normal((B, Dm) if op == "step" else (B, L, Dm))
    s = {"op": op, "cfg": cfg, "x": x, "out": torch.empty_like(x), "idx": empty((T, K), torch.int32), "gates": empty((T, K), torch.float32)}
    if op in ("forward", "backward", "step"):
        s["w"] = _layer_weights(d, c)
        s["weights"] = rb.make_weights(s["w"])
    if op == "forward":
        s["counts"] = empty((E,), torch.int32)
        s["ws"] = rb.alloc_workspace(cfg)
    elif op == "step":
        # a generation under way: states of the size that earlier tokens leave
        s["conv_state"] = d.normal32((B, D_CONV - 1, De))
        s["ssm_state"] = d.normal32((B, De, N_STATE), 0.3)
        s["ws"] = rb.alloc_workspace(cfg)
    elif op == "backward":
        s["dout"] = d.normal(x.shape)
        names = ("W_r", "W_inz", "w_conv", "b_conv", "W_x", "W_dt", "b_dt", "A", "D", "W_out") + (("b_r",) if s["w"]["b_r"] is not None else ())
        s["grads"] = {"d" + n: empty(s["w"][n].shape, torch.float32) for n in names}
        s["gstruct"] = rb.make_grads(s["grads"])
        s["ws"] = empty((rb.layer_backward_workspace_size(cfg),), torch.uint8)
    elif op == "ffn":
        # the routing decision is the preceding layer's: made here, handed to the call
        d_ff = 4 * Dm
        W_r, b_r = _router(d, c, Dm)
        route_ws = rb.alloc_workspace(cfg)
        rb.rom_route(cfg, x, W_r, b_r, s["idx"], s["gates"], None, None, None, None, route_ws)
        torch.cuda.synchronize()
        s.update(d_ff=d_ff, W_gu=d.normal((E, 2 * d_ff, Dm), Dm ** -0.5), W_down=d.normal((E, Dm, d_ff), d_ff ** -0.5),
                 ws=empty((rb.ffn_moe_workspace_size(cfg, d_ff),), torch.uint8))
    else:
        s["w"] = _mamba2_weights(d, c)
        s["weights"] = rb.make_mamba2_weights(s["w"])
        s["counts"] = empty((E,), torch.int32)
        s["ws"] = empty((rb.mamba2_workspace_size(cfg, HEADDIM),), torch.uint8)
    return s


def run(s):
    op = s["op"]
    if op == "forward":
        rb.rom_layer_forward(s["cfg"], s["weights"], s["x"], s["out"], s["idx"], s["gates"], s["counts"], s["ws"])
        return s["out"], s["idx"], s["gates"], s["counts"]
    if op == "step":
        rb.rom_layer_step(s["cfg"], s["weights"], s["x"], s["conv_state"], s["ssm_state"], s["out"], s["idx"], s["gates"], s["ws"])
        return s["out"], s["conv_state"], s["ssm_state"], s["idx"], s["gates"]
    if op == "backward":
        rb.rom_layer_backward(s["cfg"], s["weights"], s["x"], s["dout"], s["out"], s["gstruct"], s["ws"])
        return {"dx": s["out"], **s["grads"]}
    if op == "ffn":
        rb.rom_ffn_moe_forward(s["cfg"], s["d_ff"], s["W_gu"], s["W_down"], s["x"], s["idx"], s["gates"], s["out"], s["ws"])
        return s["out"]
    rb.rom_mamba2_layer_forward(s["cfg"], HEADDIM, s["weights"], s["x"], s["out"], s["idx"], s["gates"], s["counts"], s["ws"])
    return s["out"], s["idx"], s["gates"], s["counts"]


def work(case):
    c, op = case, case["op"]
    Dm, De, R = _dims(c)
    T, E, K = c["B"] * c["L"], c["E"], c["K"]
    A = T * K
    esz = 4 if c["dtype"] == "f32" else 2
    used = E * (1.0 - (1.0 - K / E) ** T)                     # experts that at least one of T tokens reaches
    io = 2 * T * Dm * esz                                     # x in, out out
    small = esz * (De * (2 * R + 2 * N_STATE + D_CONV) + E * Dm) + 4 * De * (N_STATE + 3)
    tables = 8 * A
    scan = 7.0 * T * De * N_STATE                             # decay, input, update and output of every state
    small_flops = 2.0 * T * De * (2 * R + 2 * N_STATE)
    if op == "ffn":
        d_ff = 4 * Dm
        return {"bytes": io + tables + used * 3 * d_ff * Dm * esz, "flops": 6.0 * A * Dm * d_ff}
    if op == "mamba2":
        W = 2 * De + 2 * N_STATE + De // HEADDIM
        return {"bytes": io + tables + used * (W + De) * Dm * esz + esz * E * Dm + 4 * De, "flops": 2.0 * A * Dm * (W + De) + scan}
    if op == "backward":
        # the activations are recomputed from x (input projection, conv, small projections, scan), then reversed
        weights = E * 3 * De * Dm
        return {"bytes": io + T * Dm * esz + (esz + 4) * weights + small * (1 + 4 / esz),
                "flops": 2.0 * A * Dm * De * (2 + 2 * 3) + 3 * small_flops + 4 * scan}
    state = 2 * 4 * T * De * (N_STATE + D_CONV - 1) if op == "step" else 0
    return {"bytes": io + tables + used * 3 * De * Dm * esz + small + state, "flops": 6.0 * A * Dm * De + small_flops + scan}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 1e-3}                     # fp32 sums of up to 1024 terms through four projections and a recurrence
    # activations between the stages are rounded to bf16 (2^-9 relative each): another rounding point or summation order
    # moves the result by a few of those; routing indices are decided in fp64 and stay the same
    return {"rel": 1e-2, "max": 0.1}
