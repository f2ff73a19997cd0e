"""The work that a user of this library has it do, as cases that can be timed and compared.

Five calls or call sequences of the public binding cover it:

  fused        one lossy_fused_step with drift norms: the whole lossy data-parallel step, the library's main use
  prepared     the same through lossy_fused_step_prepared, what a training loop over small fixed buffers uses
  unfused      lossy_aggregate, lossy_step, lossy_broadcast, drift_norms in turn: a program that looks at the
               estimate or clips it between the phases
  closed_loop  lossy_closed_loop_grads, then lossy_fused_step: the synthetic training run in which staleness feeds
               back into the gradients
  diagnostics  drift_pairwise and lossy_packet_sqnorms: what an experiment reads out between steps

Sizes: the bucket of one LLaMA-2-7B-shaped decoder layer and parts of it (`workload.synth.LAYER_ELEMS`), the 1 Mi
element bucket and the drop rates of the benchmark configurations, the customary 25 MiB gradient bucket, and packets of
1024 to 4096 elements (the configurations), of 256 and 512 (small ones), of 736 bf16 elements = 1472 bytes (what one
UDP datagram of an Ethernet frame carries) and of 4480 bf16 elements = 8960 bytes (the same for jumbo frames).
"""
from __future__ import annotations

import math

import torch

import paper_2507_07114_b200 as L
from workload.synth import LAYER_ELEMS

ATTENTION_ELEMS = 4 * 4096 * 4096        # q, k, v, o of a decoder layer
MLP_ELEMS = 3 * 4096 * 11008             # gate, up, down of a decoder layer
BUCKET_ELEMS = 25 * 1024 * 1024 // 2     # a 25 MiB bucket of bf16 gradients
MAX_BYTES = 15.0e9                       # a drawn case moves no more than this (the largest listed one: 17.7e9)
FIRST_STEP = 1001                        # passes are steps of a run under way


def _case(name, call, W, n, P, p, grad="bf16", replica="bf16", optimizer="adam", loss="independent", elided=False):
    return {"name": name, "call": call, "W": W, "n": n, "P": P, "p": p, "grad": grad, "replica": replica,
            "optimizer": optimizer, "loss": loss, "elided": elided}


def listed():
    return [
        # A small odd bucket (norm weights and biases of a small model): latency and launches are all of it.
        _case("small_ragged_w4_sgd_f32", "fused", 4, 100_003, 1024, 0.1, "f32", "f32", "sgd"),
        # The 1 Mi element fp32 configuration, stepped in a loop over fixed buffers.
        _case("w4_1m_sgd_f32", "prepared", 4, 1 << 20, 1024, 0.1, "f32", "f32", "sgd"),
        # One 25 MiB gradient bucket, as data-parallel wrappers cut a model: a step of about a tenth of a millisecond.
        _case("w8_25mib_bucket", "fused", 8, BUCKET_ELEMS, 2048, 0.1),
        # The headline configuration: a decoder layer, eight workers.
        _case("w8_layer", "fused", 8, LAYER_ELEMS, 2048, 0.1),
        # Many workers on a layer's attention block.
        _case("w64_attention", "fused", 64, ATTENTION_ELEMS, 4096, 0.1),
        # The sweep's hardest point: small packets at heavy loss, sixteen workers.
        _case("w16_layer_p256_heavy", "fused", 16, LAYER_ELEMS, 256, 0.3),
        # Packets as an Ethernet network has them, a layer's MLP block.
        _case("w8_mlp_ethernet", "fused", 8, MLP_ELEMS, 736, 0.1),
        # Jumbo frames, owner-elided replicas (the layout that lets a whole model fit), a bucket that ends mid-packet.
        _case("w16_jumbo_elided", "fused", 16, ATTENTION_ELEMS + 4100, 4480, 0.05, elided=True),
        # Everything in fp32, few workers, small packets.
        _case("w4_f32_adam_p512", "fused", 4, ATTENTION_ELEMS, 512, 0.1, "f32", "f32"),
        # The four phases as calls of their own on a layer's MLP block.
        _case("w8_mlp_unfused", "unfused", 8, MLP_ELEMS, 2048, 0.1),
        # The closed-loop run at its benchmark size, with losses that come in bursts.
        _case("w8_closed_loop_bursty", "closed_loop", 8, 2048 * 4096, 2048, 0.2, loss="bursty"),
        # What an experiment measures between steps: pairwise drift and the norm of every gradient piece.
        _case("w16_diagnostics", "diagnostics", 16, 4096 * 4096, 2048, 0.1),
    ]


def draw(rng):
    """Another case of the same ranges: any call, 2 to 64 workers, buckets from 50 thousand elements to a layer, packets
    from 128 elements to a jumbo frame (half of them powers of two), every loss rate, type, optimizer and option."""
    while True:
        call = rng.choice(["fused"] * 6 + ["prepared", "unfused", "unfused", "closed_loop", "diagnostics"])
        W = int(round(math.exp(rng.uniform(math.log(2), math.log(64)))))
        top = 4 << 20 if call == "prepared" else 1 << 24 if call == "diagnostics" else LAYER_ELEMS
        n = int(math.exp(rng.uniform(math.log(50_000), math.log(top))))
        if rng.random() < 0.5:
            P = 1 << rng.randint(7, 13)
        else:
            P = 8 * int(math.exp(rng.uniform(math.log(16), math.log(1120))))
        if rng.random() < 0.5:
            n -= n % P                                  # whole packets
        p = rng.choice([0.0, 0.01, 0.05, 0.1, 0.2, 0.3])
        grad, replica = rng.choice([("bf16", "bf16")] * 4 + [("f32", "f32"), ("bf16", "f32")])
        c = _case("", call, W, n, P, p, grad, replica, rng.choice(["adam", "adam", "adam", "sgd"]),
                  "bursty" if rng.random() < 0.2 else "independent", call != "closed_loop" and rng.random() < 0.2)
        del c["name"]
        if n >= P and work(c)["bytes"] <= MAX_BYTES:
            return c


def _dtype(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _rows(W, n, dtype, device):
    """W rows of n elements, each on a 256-byte boundary; the padding is zero and stays so."""
    stride = (n + 127) // 128 * 128
    base = torch.zeros(W, stride, dtype=dtype, device=device) if stride != n else torch.empty(W, n, dtype=dtype, device=device)
    return base, [base[i, :n] for i in range(W)]


def _blocks(base):
    return list(base.split(8))


class State:
    """One simulated run: the library's context, the W gradient buffers, the owners' parameters and moments, the W replicas."""

    def __init__(self, case, seed):
        c = self.case = case
        dev = torch.device("cuda", torch.cuda.current_device())
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        W, n, P, p = c["W"], c["n"], c["P"], c["p"]
        K = -(-n // P)
        call = c["call"]
        self.step = FIRST_STEP
        self.ctx, self.destroy = None, L.lossy_destroy
        gdt, rdt = _dtype(c["grad"]), _dtype(c["replica"])
        self.ctx = L.lossy_init(W=W, n=n, packet_elems=P, p_grad=p, p_param=p, seed=seed, grad_dtype=gdt, replica_dtype=rdt,
                                optimizer=c["optimizer"], lr=1e-2 if c["optimizer"] == "sgd" else 3e-4,
                                flags=L.LOSSY_REPLICA_SKIP_OWNER if c["elided"] else 0)
        if c["loss"] == "bursty":
            # bursts of four on average, the same stationary loss rate; the links start in that state
            leave = 0.25
            bits = torch.rand(2, K, W, generator=gen, device=dev) < p
            weights = torch.ones(W, dtype=torch.int64, device=dev) << torch.arange(W, device=dev)
            words = (bits * weights).sum(-1)
            self.links = torch.cat([words, words]).contiguous()
            L.lossy_set_bursty(self.ctx, p * leave / (1.0 - p), leave, self.links)
        # gradients N(0, 1e-3), parameters N(0, 0.02), moments as they are in mid-run
        self.grad_base, self.grads = _rows(W, n, gdt, dev)
        for g in self.grads:
            g.normal_(0.0, 1e-3, generator=gen)
        self.master = torch.empty(n, device=dev).normal_(0.0, 0.02, generator=gen)
        self.m = self.v = None
        if c["optimizer"] == "adam" and call != "diagnostics":
            self.m = torch.empty(n, device=dev).normal_(0.0, 1e-4, generator=gen)
            self.v = torch.empty(n, device=dev).uniform_(0.5e-7, 2e-7, generator=gen)
        self.rep_base, self.replicas = _rows(W, n, rdt, dev)
        pps = -(-K // W)
        for i, r in enumerate(self.replicas):
            lo, hi = min(n, i * pps * P), min(n, (i + 1) * pps * P)
            if c["elided"]:                              # a replica without its own shard
                r.zero_()
                r[:lo].copy_(self.master[:lo])
                r[lo:n - (hi - lo)].copy_(self.master[hi:])
            else:
                r.copy_(self.master)
        if call == "diagnostics":
            # copies of different ages: a packet that missed its broadcast is one update off
            for i, r in enumerate(self.replicas):
                old = torch.empty(n, device=dev).normal_(0.0, 3e-4, generator=gen)
                late = (torch.rand(K, generator=gen, device=dev) < p + 0.05).repeat_interleave(P)[:n]
                r.add_((old * late).to(rdt))
        self.norms = torch.zeros(W, device=dev)
        if call == "prepared":
            self.call = L.lossy_fused_step_prepared(self.ctx, self.grads, self.master, self.m, self.v, self.replicas, norms=self.norms)
        elif call == "unfused":
            self.ghat = torch.empty(n, device=dev)
            self.count = torch.empty(K, dtype=torch.uint8, device=dev)
            self.recv = torch.empty(K, dtype=torch.int64, device=dev)
            self.stale = torch.empty(K, dtype=torch.int64, device=dev)
        elif call == "closed_loop":
            self.noise_base, self.noise = self.grad_base, self.grads      # the mini-batch noise; the gradients are computed
            self.grad_base, self.grads = _rows(W, n, gdt, dev)
            self.curv = torch.empty(n, device=dev).uniform_(0.5, 1.5, generator=gen)
            self.target = torch.empty(n, device=dev).normal_(0.0, 0.02, generator=gen)
        elif call == "diagnostics":
            self.d2 = torch.empty(W * W, dtype=torch.float64, device=dev)
            self.sq = torch.empty(W * K, device=dev)

    def __del__(self):
        if self.ctx is not None:
            self.destroy(self.ctx)


def prepare(case, seed):
    return State(case, seed)


def run(s):
    call, step = s.case["call"], s.step
    s.step += 1
    if call == "diagnostics":
        s.d2.zero_()
        L.drift_pairwise(s.ctx, s.replicas, s.d2)
        L.lossy_packet_sqnorms(s.ctx, s.grads, s.sq)
        return [s.d2, s.sq]
    if call == "unfused":
        L.lossy_aggregate(s.ctx, step, s.grads, s.ghat, s.count, s.recv)
        L.lossy_step(s.ctx, step, s.ghat, s.count, s.master, s.m, s.v)
        L.lossy_broadcast(s.ctx, step, s.master, s.replicas, s.stale)
        L.drift_norms(s.ctx, s.master, s.replicas, norms=s.norms)
        return [s.ghat, s.count, s.recv, s.stale, s.master, s.m, s.v, s.norms, *_blocks(s.rep_base)]
    if call == "prepared":
        s.call(step)
    else:
        if call == "closed_loop":
            L.lossy_closed_loop_grads(s.ctx, s.curv, s.target, s.noise, s.replicas, s.grads)
        L.lossy_fused_step(s.ctx, step, s.grads, s.master, s.m, s.v, s.replicas, norms=s.norms)
    out = [s.master, s.m, s.v, s.norms, *_blocks(s.rep_base)]
    return out + _blocks(s.grad_base) if call == "closed_loop" else out


def work(case):
    """Bytes and operations of one pass: delivered gradients read, state read and written, fresh replicas written, stale
    ones read (dropped packets are neither)."""
    W, n, P, p = case["W"], case["n"], case["P"], case["p"]
    gb, rb = (2 if case[t] == "bf16" else 4 for t in ("grad", "replica"))
    adam = case["optimizer"] == "adam"
    state = 24 if adam else 8
    copies = W - 1 if case["elided"] else W
    update = 14 if adam else 2
    fused = (1 - p) * W * gb + state + copies * rb
    flops = (1 - p) * W + 1 + update + 3 * p * (W - 1)
    if case["call"] == "diagnostics":
        return {"bytes": n * (copies * rb + W * gb), "flops": n * (1.5 * W * (W - 1) + 2 * W)}
    if case["call"] == "unfused":
        fresh = (W - 1) * (1 - p) + (0 if case["elided"] else 1)
        agg, step, bcast, drift = (1 - p) * W * gb + 4, state + 4, 4 + fresh * rb, 4 + copies * rb
        return {"bytes": n * (agg + step + bcast + drift), "flops": n * ((1 - p) * W + 1 + update + 3 * copies)}
    if case["call"] == "closed_loop":
        # the gradients are written once and read once by the step
        return {"bytes": n * (8 + W * (2 * gb + rb) + fused), "flops": n * (flops + 3 * W)}
    return {"bytes": n * fused, "flops": n * flops}


def tolerance(case):
    """About four times the distance between the fp32 path and the same pass in fp64. In fp32 it is 4e-8 (m, v, estimate;
    parameters 2.5e-8) and 7e-8 for the packet norms. A bf16 value on the edge of a rounding interval may round the other way:
    2.1e-6 for replicas, 1.3e-5 for the closed loop's bf16 gradients. Counts and bit sets are whole numbers and the same."""
    if case["call"] == "closed_loop" and case["grad"] == "bf16":
        return {"rel": 5e-5}
    if case["call"] != "diagnostics" and "bf16" in (case["replica"], case["grad"] if case["call"] == "closed_loop" else ""):
        return {"rel": 1e-5}
    return {"rel": 3e-7}
