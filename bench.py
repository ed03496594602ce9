#!/usr/bin/env python
"""Benchmark of the INT4 RNN-T hot path on B200.

One step = one pass of the whole path over one batch of synthetic input: feature
prologue, input quantization, six bidirectional quantized LSTM layers, projection,
then alignment-length synchronous beam search (width 16) with density-ratio LM fusion
and the trace-back.  Default workload: the end-to-end configuration (64 utterances of
10 s, first encoder layer and joint output layer at 8 bit, everything else at 4 bit).

Prints ONE JSON line (rank 0).  `--impl reference` times the CPU oracle instead, on a
bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np

TAG_NAMES = {1: "quantize", 2: "enc_input_gemm", 3: "enc_recurrent_step", 4: "linear",
             5: "pred_lstm", 6: "pred_proj", 7: "src_lstm", 8: "src_head", 9: "tgt_lstm_l1",
             10: "tgt_lstm_l2", 11: "tgt_head", 12: "joint", 13: "beam_select", 14: "other",
             15: "search_cells", 16: "state_products"}

WORKLOADS = {
    # name: (B, T100 or T, U_max, first-layer bits, joint-out bits, has encoder, has decoder)
    "cfg4_end_to_end": dict(B=64, T=500, U_max=250, l1_bits=8, out_bits=8, enc=True, dec=True, seed=4),
    "cfg1_encoder": dict(B=32, T=500, U_max=0, l1_bits=4, out_bits=4, enc=True, dec=False, seed=1),
    "cfg3_beam": dict(B=16, T=300, U_max=150, l1_bits=4, out_bits=4, enc=False, dec=True, seed=3),
    # single unidirectional layer (K=64, H=128, B=4, T=50) and the prediction + joint networks driven
    # with drawn label sequences (256 hypothesis rows x 300 steps)
    "cfg0_single_layer": dict(B=4, T=50, U_max=0, l1_bits=4, out_bits=4, enc=False, dec=False, seed=0, kind="layer"),
    "cfg2_pred_joint": dict(B=16, T=300, U_max=0, l1_bits=4, out_bits=4, enc=False, dec=False, seed=2, kind="predjoint"),
    # the same beam workload driven time-synchronously (its wording): at most 2 labels per frame,
    # 3 calls per frame, 900 calls
    "cfg3_beam_time_synchronous": dict(B=16, T=300, U_max=150, l1_bits=4, out_bits=4, enc=False, dec=True,
                                       seed=3, tsd=2),
    # reduced lengths of the same shapes, for profiler captures that must end by themselves
    "prof_encoder": dict(B=32, T=250, U_max=0, l1_bits=4, out_bits=4, enc=True, dec=False, seed=1),
    "prof_end_to_end": dict(B=64, T=24, U_max=12, l1_bits=8, out_bits=8, enc=True, dec=True, seed=4),
    # the encoder of the end-to-end workload at a quarter of its length (64 utterances: one group of 8
    # sequences more than resident clusters, so the clusters of one direction take turns)
    "prof_encoder_64": dict(B=64, T=128, U_max=0, l1_bits=8, out_bits=4, enc=True, dec=False, seed=4),
    # the regime of the paper's run-time figure (Section 4.1): ONE utterance of 152 encoder frames,
    # everything at 4 bits, beam width from --beam (1..16): 16 hypothesis rows at most, so every
    # step streams all weights for a handful of rows
    "fig2_single_utterance": dict(B=1, T=152, U_max=76, l1_bits=4, out_bits=4, enc=True, dec=True, seed=6),
    # the same utterance with the precision assignment of the end-to-end workload (first encoder layer
    # and joint output layer at 8 bits, the rest at 4): the "mixed" point of that figure
    "fig2_single_utterance_mixed": dict(B=1, T=152, U_max=76, l1_bits=8, out_bits=8, enc=True, dec=True, seed=6),
    # and with every weight and every activation quantizer at 8 bits: the "INT8" bar of that figure
    "fig2_single_utterance_int8": dict(B=1, T=152, U_max=76, l1_bits=8, out_bits=8, enc=True, dec=True, seed=6,
                                       all8=True),
}


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return dict(hbm_gbs=d["hbm_gbs"], bf16_tflops=d["bf16_tflops"],
                    bf16_tflops_sustained=d.get("bf16_tflops_sustained", d["bf16_tflops"]),
                    source="measured")
    return dict(hbm_gbs=6650.0, bf16_tflops=1590.0, bf16_tflops_sustained=1400.0, source="fallback")


class ClockSampler:
    """nvidia-smi clock / throttle-reason samples during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.p = None
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                       "-i", str(gpu_index), "-lms", "50"], stdout=self.f,
                                      stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None

    def stop(self):
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        if self.p is None:
            return out
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except Exception:
            self.p.kill()
        self.f.flush()
        self.f.seek(0)
        sm, mx, reasons = [], [], set()
        for line in self.f.read().splitlines():
            c = [x.strip() for x in line.split(",")]
            if len(c) < 9:
                continue
            try:
                sm.append(float(c[1]))
                mx.append(float(c[2]))
            except ValueError:
                continue
            for name, v in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), c[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        try:
            os.unlink(self.f.name)
        except OSError:
            pass
        if sm:
            busy = [v for v in sm if v >= 0.5 * max(sm)] or sm
            out.update(sm_mhz=statistics.median(busy), sm_max_mhz=max(mx), reasons=sorted(reasons),
                       samples=len(sm))
        return out


# ------------------------------------------------------------------------------------ oracle arm
def oracle_sample(wl_name: str, cores: int, frames: int = 8):
    """The CPU oracle on a bounded sample of the workload: `cores` utterances cut to the first
    `frames` encoder frames (2*frames log-mel frames), label budget frames/2, all layers at
    full width.  Returns (seconds, audio_seconds, description)."""
    from oracle import oracle as O
    from paper_2206_07882_b200 import synth
    wl = WORKLOADS[wl_name]
    n = max(1, cores)
    seed = wl["seed"]
    t0 = time.perf_counter()
    e = None
    kind = wl.get("kind", "rnnt")
    if kind == "layer":      # the whole workload: the oracle finishes it in well under a second
        w = synth.single_layer(seed=seed, T=wl["T"], B=wl["B"])
        xa, ha = O.act_symmetric(w["x_clip"], 4), O.act_symmetric(1.0, 4)
        t0 = time.perf_counter()
        O.lstm_layer(O.Lstm(w["layers"]), O.quantize(w["x"], xa), xa, ha, n_threads=n)
        dt = time.perf_counter() - t0
        return dt, wl["B"] * wl["T"] * 0.02, f"the whole workload ({wl['B']} sequences x {wl['T']} steps)"
    if kind == "predjoint":  # `cores` of the 256 rows over the first 4 * frames steps
        steps = 4 * frames
        dw = synth.decoder(seed)
        act = O.act_symmetric(1.0, 4)
        fr = synth.enc_frames(seed, steps, 1, 1280).astype(np.float32)
        proj = synth._linear(synth.Stream(seed), "enc.proj", 256, 1280)
        toks = np.concatenate([np.zeros((n, 1), np.int32), synth.labels(seed, n, steps - 1, 1024)], axis=1)
        fi = np.tile(np.arange(steps, dtype=np.int32)[None, :], (n, 1))
        dec = O.Decoder(dw)
        t0 = time.perf_counter()
        e = O.linear(O.Linear(proj), O.quantize(fr.reshape(steps, 1280), act), act)
        O.pred_joint_forced(dec, e, fi, toks, n_threads=n)
        dt = time.perf_counter() - t0
        # scaled to the unit of the line: seconds per second of "audio" at 16 rows per utterance
        return dt, n * steps * 0.02 / 16.0, f"{n} of the 256 rows x first {steps} of 300 steps, full layer widths, one row per thread"
    if wl["enc"]:
        enc_w = synth.encoder(seed, T=frames, B=n, first_layer_bits=wl["l1_bits"], in_max=wl["l1_bits"] == 8,
                              features=False)
        if wl_name.startswith("cfg4"):
            mel = synth.logmel(seed, n, 2 * frames, 40)
            feats = np.stack([O.features(mel[b]) for b in range(n)], axis=1).astype(np.float16)
        else:
            feats = synth.Stream(seed).normal("features", (frames, n, 240)).astype(np.float16)
        e = O.encoder_forward(enc_w["enc"], feats, n_threads=n)["e"]
    if wl["dec"]:
        u = max(1, frames // 2)
        dw = synth.decoder(3, out_bits=wl["out_bits"], U_max=u)
        if e is None:
            act = O.act_symmetric(1.0, 4)
            fr = synth.enc_frames(seed, frames, n, 1280).astype(np.float32)
            proj = synth._linear(synth.Stream(seed), "enc.proj", 256, 1280)
            e = O.linear(O.Linear(proj), O.quantize(fr.reshape(frames * n, 1280), act), act).reshape(frames, n, 256)
        O.alsd(O.Decoder(dw), e, trace=False, n_threads=n)
    dt = time.perf_counter() - t0
    audio = n * frames * 0.02
    what = (f"{n} utterances x first {frames} encoder frames ({audio:.2f} s of audio), label budget "
            f"{max(1, frames // 2)}, full layer widths, one utterance per thread")
    return dt, audio, what


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cores = min(os.cpu_count() or 1, 8)
    from oracle import oracle as O
    O.build()
    times = []
    what = ""
    audio = 1.0
    for i in range(args.warmup + args.steps):
        dt, audio, what = oracle_sample(args.workload, cores, frames=args.ref_frames)
        if i >= args.warmup:
            times.append(dt)
    t = sum(times) / len(times)
    rtf = t / audio
    line = {"impl": "reference", "metric": "end_to_end_rtf", "value": rtf, "unit": "s/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup, "ms_per_step": t * 1e3,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int4",
            "data": "synthetic", "config": {"workload": args.workload, "sample": what},
            "cpu_baseline": {"value": rtf, "unit": "s/s", "cores": cores, "kind": "oracle", "sample": what},
            "e2e": {"value": rtf, "unit": "s/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------------------------ GPU arm
class Job:
    """Holds device weights and buffers of one workload and runs whole steps."""

    def __init__(self, wl_name: str, rank: int, beam: int = 16, groups: int = 1):
        import torch
        from paper_2206_07882_b200 import binding as Bd
        from paper_2206_07882_b200 import synth
        self.torch, self.Bd = torch, Bd
        wl = self.wl = WORKLOADS[wl_name]
        self.name = wl_name
        self.W = max(1, min(16, beam))
        B, T = wl["B"], wl["T"]
        from paper_2206_07882_b200 import sharding
        seed = sharding.rank_seed(wl["seed"], rank)    # every rank gets its own utterances
        self.enc = self.dec = None
        self.host_in = None
        self.kind = wl.get("kind", "rnnt")
        if self.kind == "layer":
            w = synth.single_layer(seed=wl["seed"], T=T, B=B)
            self.layer = [Bd.DeviceLstm(l) for l in w["layers"]]
            self.layer_act = Bd.q4_act_symmetric(w["x_clip"], 4)
            self.host_in = torch.from_numpy(synth.single_layer(seed=seed, T=T, B=B)["x"].reshape(T * B, -1)).pin_memory()
            self.layer_ws = None
        if self.kind == "predjoint":
            dw = synth.decoder(wl["seed"])
            self.pj = Bd.Decoder(dw)
            # one-time int8 operands: with them the library runs these calls on the tensor cores
            self.pj.pred_lstm.prepare()
            self.pj.pred_proj.prepare()
            self.pj.joint_out.prepare()
            N = B * 16
            self.pj_tok = torch.from_numpy(np.ascontiguousarray(np.concatenate(
                [np.zeros((N, 1), np.int32), synth.labels(seed, N, T - 1, 1024)], axis=1).T)).cuda()   # [T, N]
            self.pj_fi = torch.from_numpy((np.arange(T, dtype=np.int32)[:, None] * B +
                                           (np.arange(N, dtype=np.int32)[None, :] // 16)).astype(np.int32)).cuda()
            self.host_in = torch.from_numpy(synth.enc_frames(seed, T, B, 1280)).pin_memory()
            self.frame_act = Bd.q4_act_symmetric(1.0, 4)
            self.frame_proj = Bd.DeviceLinear(synth._linear(synth.Stream(wl["seed"]), "enc.proj", 256, 1280)).prepare()
            Hp = self.pj.pred_lstm.H
            self.pj_buf = dict(hq=[torch.zeros((N, Hp // 2), dtype=torch.uint8, device="cuda") for _ in range(2)],
                               c=torch.zeros((N, Hp), dtype=torch.float32, device="cuda"),
                               logp=torch.empty((N, 1024), dtype=torch.float32, device="cuda"),
                               ws=torch.empty(Bd.workspace_bytes(Bd.WS_JOINT, [N, 256, Hp]), dtype=torch.uint8, device="cuda"))
        if wl["enc"]:
            a8 = 8 if wl.get("all8") else 4
            enc_w = synth.encoder(wl["seed"], T=T, B=B, first_layer_bits=wl["l1_bits"],
                                  in_max=wl["l1_bits"] == 8, features=False, layer_bits=a8, proj_bits=a8)
            self.enc = Bd.Encoder(enc_w["enc"])
            if wl_name.startswith("cfg4"):
                self.host_in = torch.from_numpy(synth.logmel(seed, B, 2 * T, 40)).pin_memory()
            else:
                self.host_in = torch.from_numpy(
                    synth.Stream(seed).normal("features", (T, B, 240)).astype(np.float16)).pin_memory()
        if wl["dec"]:
            dw = synth.decoder(3, out_bits=wl["out_bits"], U_max=wl["U_max"], all_bits=8 if wl.get("all8") else 4)
            # optionally the batch is searched as `groups` sets side by side (same weights, separate states
            # and streams)
            self.groups = groups if (groups > 1 and B >= 32 and "tsd" not in wl) else 1
            self.dec = Bd.GroupedDecoder(dw, self.groups) if self.groups > 1 else Bd.Decoder(dw)
            if "tsd" in wl:
                self.dec.alloc_state(B, self.W, T * (wl["tsd"] + 1), wl["tsd"])
            else:
                self.dec.alloc_state(B, self.W, T + wl["U_max"])
            if not wl["enc"]:
                self.host_in = torch.from_numpy(synth.enc_frames(seed, T, B, 1280)).pin_memory()
                self.frame_act = Bd.q4_act_symmetric(1.0, 4)
                self.frame_proj = Bd.DeviceLinear(synth._linear(synth.Stream(wl["seed"]), "enc.proj", 256, 1280)).prepare()
        self.dev_in = self.host_in.cuda()
        self.graph = None

    def step_graphed(self, mark=None):
        """The same pass over self.dev_in, replayed as two CUDA graphs (encoder side, search
        side) so that one event between them splits the step time."""
        if self.graph is None:
            self._e = None

            def enc_part():
                self._e = self.encode(self.dev_in)
                return self._e

            self.graph = [self.Bd.GraphedStep(enc_part), None]
            self.graph[0]()
            self.graph[1] = self.Bd.GraphedStep(lambda: self.search(self.graph[0].result))
        if mark:
            mark("start")
        self.graph[0]()
        if mark:
            mark("encoded")
        res = self.graph[1]()
        if mark:
            mark("decoded")
        return res

    def h2d_bytes(self):
        return self.host_in.numel() * self.host_in.element_size()

    def encode(self, x):
        """Encoder side of a pass: returns (projected frames e [T,B,D], last result so far)."""
        Bd, wl = self.Bd, self.wl
        B, T = wl["B"], wl["T"]
        if self.kind == "layer":
            xq = Bd.quantize_pack_int4(x, self.layer_act)
            r = Bd.qlstm_layer_forward(xq, self.layer_act, T, B, self.layer, workspace=self.layer_ws)
            self.layer_ws = r["workspace"]
            return None, r["yq"]
        if self.enc is not None:
            feats = Bd.q4_feature_prologue(x) if self.name.startswith("cfg4") else x
            r = self.enc.forward(feats)
            return r["e"], r["yq"]
        fq = Bd.quantize_pack_int4(x.reshape(T * B, 1280), self.frame_act)
        return Bd.q4_linear_forward(fq, self.frame_act, self.frame_proj).reshape(T, B, 256), None

    def search(self, enc_out):
        e, res = enc_out if isinstance(enc_out, tuple) else (enc_out, None)
        if self.kind == "predjoint":
            # teacher-forced prediction network + joint: every step feeds the drawn label of each of the
            # 256 rows (embedding lookup inside qlstm_step), then scores the row against its frame
            Bd, d, b = self.Bd, self.pj, self.pj_buf
            b["hq"][0].zero_()
            b["c"].zero_()
            e2 = e.reshape(-1, 256)
            for s in range(self.wl["T"]):
                Bd.qlstm_step(d.pred_emb_q, d.pred_emb_act, b["hq"][s & 1], b["c"], d.pred_lstm,
                              x_row_idx=self.pj_tok[s], out=dict(hq=b["hq"][(s + 1) & 1], c=b["c"]))
                Bd.qjoint_logprobs(e2, self.pj_fi[s], b["hq"][(s + 1) & 1], d.pred_lstm.hid_act, d.pred_proj,
                                   d.z_act, d.joint_out, logp=b["logp"], workspace=b["ws"])
            return (b["logp"],)
        if self.dec is not None:
            if "tsd" in self.wl:
                res = self.dec.decode_time_synchronous(e, self.wl["tsd"], u_max=self.wl["U_max"], W=self.W)
            else:
                res = self.dec.decode(e, u_max=self.wl["U_max"], W=self.W)
        return res

    def step(self, x, mark=None):
        """One pass over device-resident input x.  mark(name) records phase boundaries."""
        if mark:
            mark("start")
        enc_out = self.encode(x)
        if mark:
            mark("encoded")
        res = self.search(enc_out)
        if mark:
            mark("decoded")
        return res

    def result_to_host(self, res):
        if isinstance(res, tuple):
            out = [t.cpu() for t in res]
            return sum(t.numel() * t.element_size() for t in out)
        # encoder-only workload: the result is the packed last-layer codes; read a checksum row
        o = res[-1].cpu()
        return o.numel() * o.element_size()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="cfg4_end_to_end", choices=sorted(WORKLOADS))
    ap.add_argument("--ref-frames", type=int, default=8)
    ap.add_argument("--beam", type=int, default=16, help="beam width W (1..16)")
    ap.add_argument("--groups", type=int, default=1,
                    help="sets of utterances searched side by side on their own streams (batches of 32 "
                         "utterances and more); measured: no gain over one set, hence 1")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sweep", action="store_true",
                    help="skip the single-utterance beam sweep appended to the end-to-end line")
    ap.add_argument("--no-dependent-launch", action="store_true",
                    help="launch the beam step's kernels in plain stream order")
    ap.add_argument("--eager", action="store_true",
                    help="launch every kernel from the host instead of replaying a CUDA graph")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
        return

    import ctypes as C
    import torch
    import torch.distributed as dist
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the library has no CPU path")
    torch.cuda.set_device(local)
    if world > 1:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    from paper_2206_07882_b200 import binding as Bd
    lib = Bd.lib()
    if args.no_dependent_launch:
        from paper_2206_07882_b200 import binding as _Bd
        _Bd.dependent_launch_set(False)
    job = Job(args.workload, rank, args.beam, args.groups)
    job.passes = args.steps
    wl = job.wl
    B, T, U = wl["B"], wl["T"], wl["U_max"]
    iters = (T * (wl["tsd"] + 1) if "tsd" in wl else T + U) if wl["dec"] else 0
    W = max(args.warmup, 3)
    K = args.steps
    use_graph = not args.eager
    run = (lambda: job.step_graphed()) if use_graph else (lambda: job.step(job.dev_in))

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    def events(n):
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(2 * n)]
        for ev in evs:
            ev.record()                      # materialise the handles
        torch.cuda.synchronize()
        return evs, (C.c_void_p * n)(*[ev.cuda_event for ev in evs[:n]]), \
            (C.c_void_p * n)(*[ev.cuda_event for ev in evs[n:]]), (C.c_int32 * n)()

    job.step(job.dev_in)                     # eager first pass: configures every kernel
    for _ in range(W):
        run()
    barrier()

    # ---- timed region 1: inputs resident in HBM
    sampler = ClockSampler(local) if rank == 0 else None
    barrier()
    l0 = Bd.launch_count()
    t_start = torch.cuda.Event(enable_timing=True)
    t_stop = torch.cuda.Event(enable_timing=True)
    tmarks = []

    def tmark(name):
        ev = torch.cuda.Event(enable_timing=True)
        ev.record()
        tmarks.append(ev)

    t_start.record()
    for _ in range(K):
        if use_graph:
            job.step_graphed(tmark)
        else:
            job.step(job.dev_in, tmark)
    t_stop.record()
    barrier()
    clocks = sampler.stop() if sampler else None
    ms_total = t_start.elapsed_time(t_stop)
    enc_ms = sum(tmarks[i].elapsed_time(tmarks[i + 1]) for i in range(0, len(tmarks), 3)) / K
    dec_ms = sum(tmarks[i + 1].elapsed_time(tmarks[i + 2]) for i in range(0, len(tmarks), 3)) / K
    per_step = sorted(tmarks[i].elapsed_time(tmarks[i + 2]) for i in range(0, len(tmarks), 3))   # each step by itself

    # ---- timed region 2: end to end through the public API with host buffers
    barrier()
    e_start = torch.cuda.Event(enable_timing=True)
    e_stop = torch.cuda.Event(enable_timing=True)
    d2h = 0
    e_start.record()
    for _ in range(K):
        if use_graph:
            job.dev_in.copy_(job.host_in, non_blocking=True)
            res = run()
        else:
            res = job.step(job.host_in.to("cuda", non_blocking=True))
        d2h = job.result_to_host(res)
    e_stop.record()
    barrier()
    ms_e2e = e_start.elapsed_time(e_stop)

    # ---- instrumented eager passes (rank 0): every launch of the pass bracketed by CUDA
    # events on its own stream -> per-kernel shares, the dominant kernel's launch duration,
    # the encoder / search split, and the number of launches per pass
    shares, dom_tag, dom_ms, dom_n, n_launch_step, rec_extra, series = {}, None, None, 0, 0, None, {}
    if rank == 0:
        cap = 40000
        evs, start, stop, tags = events(cap)
        marks = []

        def mark(name):
            ev = torch.cuda.Event(enable_timing=True)
            ev.record()
            marks.append(ev)

        # per-kernel durations are taken with the three search chains serialised on one stream
        # (auxiliary streams withdrawn for these passes), so that an event pair brackets one
        # kernel running alone, as in the profiler's launch list
        saved_aux = None
        parts = list(getattr(job.dec, "parts", [job.dec])) if job.dec is not None else []
        if parts and parts[0].state is not None:
            saved_aux = [(p.state.aux_stream[0], p.state.aux_stream[1]) for p in parts]
            for p in parts:
                p.state.aux_stream[0], p.state.aux_stream[1] = None, None
        tot, cnt, series = {}, {}, {}
        for _ in range(K):
            lib.q4_timing_set(C.c_uint32(0xFFFFFFFF), start, stop, tags, C.c_int32(cap))
            la = Bd.launch_count()
            job.step(job.dev_in, mark)
            torch.cuda.synchronize()
            n_launch_step = Bd.launch_count() - la
            n = lib.q4_timing_count()
            lib.q4_timing_set(C.c_uint32(0), None, None, None, C.c_int32(0))
            per_pass = {}
            for i in range(n):
                ms = evs[i].elapsed_time(evs[cap + i])
                tot[tags[i]] = tot.get(tags[i], 0.0) + ms
                cnt[tags[i]] = cnt.get(tags[i], 0) + 1
                per_pass.setdefault(tags[i], []).append(ms)
            for t_, v_ in per_pass.items():          # launch-ordered durations, one list per pass
                series.setdefault(t_, []).append(v_)
        if saved_aux is not None:
            for p, sv in zip(parts, saved_aux):
                p.state.aux_stream[0], p.state.aux_stream[1] = sv
        # the replayed search ends its steps with the last label, the instrumented pass runs all of them
        if use_graph and len(parts) == 1 and "tsd" not in wl and parts[0].search_plan_info()["built"]:
            run()
            torch.cuda.synchronize()
            per_step_launches = sum(cnt.get(t, 0) for t in (5, 6, 7, 8, 9, 10, 11, 12, 13, 15, 16)) / K / iters
            per_step_launches += (cnt.get(14, 0) / K) // iters               # the gather, where a step has one
            n_launch_step -= round((iters - parts[0].search_steps_taken()) * per_step_launches) - 3
        allms = sum(tot.values()) or 1.0
        shares = {TAG_NAMES.get(t, str(t)): {"launches": cnt[t] // K, "ms": round(tot[t] / K, 3),
                                             "avg_us": round(1e3 * tot[t] / cnt[t], 2),
                                             "share": round(tot[t] / allms, 4)} for t in sorted(tot)}
        # The roofline entry describes the dominant KERNEL (launch sites grouped by the kernel
        # function they launch: the fused LSTM step serves tags 5, 7, 9 and 10), and of that
        # kernel the launch site with the largest time; the encoder recurrence is reported beside
        # it when it is not the dominant one.
        families = {"k_mma_lstm": (5, 7, 9, 10), "k_enc_recurrent": (3,), "k_mma_gemm": (2,), "joint": (12,)}
        fam_ms = {f: sum(tot.get(t, 0.0) for t in ts) for f, ts in families.items()}
        dom_tag = None
        if any(v > 0 for v in fam_ms.values()):
            dom_fam = max(fam_ms, key=lambda f: fam_ms[f])
            dom_tag = max((t for t in families[dom_fam] if t in tot), key=lambda t: tot[t])
        elif tot:
            dom_tag = max(tot, key=lambda t: tot[t])
        dom_ms, dom_n = (tot[dom_tag] / cnt[dom_tag], cnt[dom_tag]) if dom_tag is not None else (0.0, 0)
        rec_extra = (tot[3] / cnt[3], cnt[3]) if 3 in tot and dom_tag != 3 else None
    barrier()

    from paper_2206_07882_b200 import sharding
    ms_total = sharding.job_time_ms(ms_total, "cuda")       # max over ranks
    ms_e2e = sharding.job_time_ms(ms_e2e, "cuda")
    ms_step = ms_total / K
    rtf = sharding.aggregate_rtf(ms_step, B, T * 0.02, world, "cuda")
    rtf_e2e = sharding.aggregate_rtf(ms_e2e / K, B, T * 0.02, world, "cuda")

    if rank == 0:
        pk = peaks()
        line = {"metric": "end_to_end_rtf", "value": rtf, "unit": "s/s", "n_gpus": world, "steps": K,
                "warmup": W, "ms_per_step": ms_step, "higher_is_better": False, "scaling": "weak",
                "ms_per_step_best": per_step[0] if per_step else None,
                "ms_per_step_median": statistics.median(per_step) if per_step else None,
                "vs_baseline": None, "dtype": "int4/int8 codes, int32 accumulate, fp32 gates",
                "data": "synthetic",
                "config": {"workload": args.workload, "utterances_per_gpu": B, "frames": T,
                           "beam": job.W if wl["dec"] else 0, "label_budget": U, "search_iterations": iters,
                           "launch": "cuda graph replay of the whole pass" if use_graph else "eager",
                           "l2": "no flush: one pass streams more than 1 GB of accumulators, codes and "
                                 "state through the 126 MB L2 between two uses of any input"},
                "parts": {"encoder_ms": enc_ms, "decode_ms": dec_ms,
                          "encoder_frames_per_s": (B * T / (enc_ms / 1e3)) if wl["enc"] and enc_ms else None,
                          "beam_hyps_per_s": (B * job.W * iters / (dec_ms / 1e3)) if wl["dec"] and dec_ms else None,
                          "layer_frames_per_s": (B * T / (enc_ms / 1e3)) if job.kind == "layer" and enc_ms else None,
                          "pred_joint_hyps_per_s": (B * 16 * T / (dec_ms / 1e3)) if job.kind == "predjoint" and dec_ms else None},
                "e2e": {"value": rtf_e2e, "unit": "s/s", "h2d_bytes_per_step": job.h2d_bytes(),
                        "d2h_bytes_per_step": d2h},
                "gpu_launches": n_launch_step * K, "launches_per_step": n_launch_step, "kernels": shares,
                "kernels_note": "eager passes with every search step; the replayed search ends its steps with the last label "
                                "and carries the iterations that are left out in two launches",
                "clocks": clocks, "peaks": pk,
                "paper_context": {"rtf_int4_simulated": 0.065, "speedup_fp16_to_int4_simulated": 3.4,
                                  "note": "simulated accelerator, 1 utterance of 152 frames, beam 16"}}
        pk["int8_tops_yardstick"] = int8_yardstick(torch)
        line["roofline"] = roofline(job, dom_tag, dom_ms, dom_n, pk, series.get(dom_tag)) if dom_tag is not None else None
        if rec_extra is not None:
            line["roofline_encoder_recurrence"] = roofline(job, 3, rec_extra[0], rec_extra[1], pk)
        if wl["dec"] and "tsd" not in wl:
            line["parts"].update(search_regimes(job, dec_ms, torch))
        if args.workload == "cfg4_end_to_end" and world == 1 and not args.no_sweep:
            line["fig2_beam_sweep"] = fig2_sweep(torch)
        if line["roofline"] is not None:
            line["roofline"]["timing"] = ("CUDA events around every launch of this kernel in eager, single-stream "
                                          "passes of the same step; the headline region replays CUDA graphs, "
                                          "inside which single launches cannot be bracketed")
        if not args.no_cpu_baseline:
            from oracle import oracle as O
            O.build()
            cores = min(os.cpu_count() or 1, 8)
            # once per run: twice the frames of a step of the reference arm (10 - 20 s of CPU work at the default)
            dt, audio, what = oracle_sample(args.workload, cores, frames=2 * args.ref_frames)
            line["cpu_baseline"] = {"value": dt / audio, "unit": "s/s", "cores": cores, "kind": "oracle",
                                    "sample": what, "seconds": dt}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


# dram__bytes_read.sum + dram__bytes_write.sum of ONE launch, copied by hand from an ncu capture of
# the kernel revision named in "captured"; None once the kernel has changed since.  The capture runs
# with cold caches; inside the timed loop the weights of an iteration stay in the L2, so the real
# DRAM traffic of a launch is lower.
NCU_TRAFFIC = {
    # target-LM layer 2 at 1024 rows, cold caches (tiles without work leave before their set-up)
    "k_mma_lstm_tgt_l2": {"bytes": 41242880 + 861952, "rows": 1024, "weights": 2 * 8192 * 2048,
                          "captured": "ncu capture of k_mma_lstm at 1024 rows, workload prof_end_to_end, cold caches; "
                                      "row-dependent part scaled to the timed rows"},
    # register-resident recurrence, one layer of 250 steps x 32 sequences
    "k_enc_recurrent": {"bytes": 167230720 + 6221056, "steps": 250, "sequences": 32,
                        "captured": "ncu capture of k_enc_recurrent_few<20,10>, workload prof_encoder; scaled by steps x "
                                    "sequences (accumulators read once, codes written once)"},
    # the same with one group of sequences more than clusters (clusters take turns), 128 steps x 64 sequences
    "k_enc_recurrent_turns": {"bytes": 171157760 + 6593792, "steps": 128, "sequences": 64,
                              "captured": "ncu capture of k_enc_recurrent_w4s<20,0>, workload prof_encoder_64; scaled by "
                                          "steps x sequences (accumulators read once, codes written once)"},
}


def int8_yardstick(torch):
    """Dense int8 GEMM rate of the library routine torch._int_mm at 8192^3, measured in this run as a
    yardstick for the int8 tensor peak (never on the timed path).  TOP/s, or None if unavailable."""
    try:
        a = torch.randint(-8, 8, (8192, 8192), dtype=torch.int8, device="cuda")
        b = torch.randint(-8, 8, (8192, 8192), dtype=torch.int8, device="cuda")
        for _ in range(3):
            torch._int_mm(a, b)
        best = None
        for _ in range(10):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            torch._int_mm(a, b)
            e1.record()
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            best = ms if best is None else min(best, ms)
        return 2.0 * 8192 ** 3 / (best / 1e3) / 1e12
    except Exception:
        return None


def search_regimes(job, dec_ms, torch):
    """Splits the search time into its two kinds of iterations.  With the synthetic weights an
    iteration either extends (nearly) every slot by a label, so that the next one runs all three
    networks on those rows, or extends none (label budgets spent: only the joint network and the
    selection run).  The label-free kind, which a search carries out together at its end, is timed by itself: the
    same search with a label budget of zero, replayed as a CUDA graph; the other kind follows from the measured search time."""
    wl, d = job.wl, job.dec
    T, B, W = wl["T"], wl["B"], job.W
    iters = T + wl["U_max"]
    tok = (d.history("bp_token") if hasattr(d, "parts") else d.tensors["bp_token"])[:iters]
    per_iter = (tok > 0).reshape(iters, -1).sum(1)
    n_busy = int((per_iter > 0).sum().item()) + 1          # launch 0 advances the start symbols
    n_free = iters - n_busy
    e = job.graph[0].result[0] if job.graph is not None else job.encode(job.dev_in)[0]
    g = job.Bd.GraphedStep(lambda: d.decode(e, u_max=0, W=W))
    g()
    g()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(3):
        g()
    e1.record()
    torch.cuda.synchronize()
    free_us = e0.elapsed_time(e1) / 3 * 1e3 / T
    busy_us = (dec_ms * 1e3 - n_free * free_us) / max(n_busy, 1)
    return {"iterations_with_network_rows": n_busy, "iterations_label_free": n_free,
            "us_per_iteration_with_network_rows": busy_us, "us_per_iteration_label_free": free_us,
            "hyps_per_s_with_network_rows": B * W / (busy_us * 1e-6) if busy_us > 0 else None,
            "hyps_per_s_label_free": B * W / (free_us * 1e-6)}


def fig2_sweep(torch):
    """The regime of the paper's run-time figure (Section 4.1): ONE utterance of 152 encoder frames,
    beam width 1..16, everything at 4 bits; ms per utterance (graph replay, inputs resident)."""
    out = {}
    job = Job("fig2_single_utterance", 0, 16)
    for W in (1, 2, 4, 8, 16):
        job.W = W
        job.dec.alloc_state(job.wl["B"], W, job.wl["T"] + job.wl["U_max"])
        job.graph = None
        job.step(job.dev_in)
        for _ in range(3):
            job.step_graphed()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(5):
            job.step_graphed()
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / 5
        out[str(W)] = {"ms_per_utterance": ms, "rtf": ms / 1e3 / (job.wl["T"] * 0.02)}
    # the precision axis of the same figure at beam 16 (the paper's simulated accelerator: RTF 0.116 all
    # 8 bit, 0.065 all 4 bit)
    for name, key in (("fig2_single_utterance_int8", "all_int8_beam16"), ("fig2_single_utterance_mixed", "mixed_beam16")):
        del job
        torch.cuda.empty_cache()
        job = Job(name, 0, 16)
        job.step(job.dev_in)
        for _ in range(3):
            job.step_graphed()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(5):
            job.step_graphed()
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / 5
        out[key] = {"ms_per_utterance": ms, "rtf": ms / 1e3 / (job.wl["T"] * 0.02)}
    return out


def roofline(job, tag, ms, n, pk, series=None):
    """Roofline entry of one kernel.  Algorithmic work per launch: the weight bytes the kernel must
    read once plus per-row state traffic, and 2*rows*J*K integer ops.  `series`: the launch-ordered
    event durations (ms) of this launch site, one list per instrumented pass."""
    name = TAG_NAMES[tag]
    wl = job.wl
    int8_peak = 2.0 * pk["bf16_tflops_sustained"]          # dense int8 : bf16 = 2 : 1 (nominal ratio)
    tensor_unit = "TOP/s (int8; peak = 2 x measured sustained bf16)"
    out = {"kernel": name, "launches_timed": n, "avg_ms": ms, "traffic": None,
           "traffic_note": "no ncu capture of the current kernel revision", "peak_source": pk["source"]}

    def entry(bytes_, ops, sec):
        t_hbm = bytes_ / (pk["hbm_gbs"] * 1e9)
        t_tensor = ops / (int8_peak * 1e12)
        r = {"algorithmic_bytes": bytes_, "algorithmic_ops": ops,
             "hbm": {"achieved": bytes_ / sec / 1e9, "peak": pk["hbm_gbs"], "unit": "GB/s",
                     "frac": bytes_ / sec / 1e9 / pk["hbm_gbs"]},
             "tensor": {"achieved": ops / sec / 1e12, "peak": int8_peak, "unit": tensor_unit,
                        "frac": ops / sec / 1e12 / int8_peak,
                        "peak_measured_int8_yardstick": pk.get("int8_tops_yardstick")}}
        if t_tensor > t_hbm:
            r.update(bound="tensor", achieved=ops / sec / 1e12, peak=int8_peak, unit="TFLOP/s",
                     frac=ops / sec / 1e12 / int8_peak)
        else:
            r.update(bound="hbm", achieved=bytes_ / sec / 1e9, peak=pk["hbm_gbs"], unit="GB/s",
                     frac=bytes_ / sec / 1e9 / pk["hbm_gbs"])
        return r

    def lstm_work(l, rows, kx):
        # weights as stored (packed codes + row scales + bias), per row: input codes, previous
        # and new cell-output codes, cell state read and written
        H = l.H
        wbytes = l.w_ih.q.numel() + l.w_hh.q.numel() + 2 * 4 * 4 * H + 4 * 4 * H
        per_row = kx * l.w_ih.bits // 8 + H * l.w_hh.bits // 8 * 2 + H * 4 * 2
        ops = 2.0 * rows * 4 * H * (l.w_ih.k_pad + H)
        return wbytes + rows * per_row, ops

    if job.dec is not None and tag in (5, 7, 9, 10):
        d = job.dec
        l, kx = {5: (d.pred_lstm, 256), 7: (d.src.lstm[0], 256), 9: (d.tgt.lstm[0], 256),
                 10: (d.tgt.lstm[-1], d.tgt.lstm[0].H)}[tag]
        # rows a launch really advances: the label extensions of the previous selection (blank
        # extensions keep their parent's state), counted from the search history of the last pass;
        # launch 0 advances the start symbol of every utterance
        iters = wl["T"] * (wl["tsd"] + 1) if "tsd" in wl else wl["T"] + wl["U_max"]
        # (with the batch searched as several sets, a launch serves one set: launches come in
        # iteration-major order, one per set)
        parts = list(getattr(job.dec, "parts", [job.dec]))
        cols = []
        for p_ in parts:
            tk = p_.tensors["bp_token"][:iters]
            pi = (tk > 0).reshape(iters, -1).sum(1).cpu().numpy().astype(np.float64)
            cols.append(np.concatenate([[float(p_.B)], pi[:-1]]))
        rows = np.stack(cols, axis=1).reshape(-1)
        iters = iters * len(parts)
        busy = rows > 0
        mean_rows = float(rows.mean())
        out.update(rows_per_launch_mean=mean_rows, launches_with_rows=int(busy.sum()),
                   launches_without_rows=int((~busy).sum()), mean_rows_when_any=float(rows[busy].mean()))
        times = None
        if series and all(len(v) == iters for v in series):
            times = np.asarray(series, dtype=np.float64)            # [passes, launches]
        if times is not None and busy.any():
            # the headline fraction describes the launches that HAVE rows (ops at their mean row count
            # over their mean duration); the all-launch mean, which mixes them with launches that find
            # no pending row and exit at once, is kept beside it
            ms_busy = float(times[:, busy].mean())
            b_, o_ = lstm_work(l, float(rows[busy].mean()), kx)
            out.update(entry(b_, o_, ms_busy / 1e3))
            out["avg_ms_with_rows"] = ms_busy
            out["avg_ms_without_rows"] = float(times[:, ~busy].mean()) if (~busy).any() else None
            b2, o2 = lstm_work(l, mean_rows, kx)
            out["frac_mean"] = entry(b2, o2, ms / 1e3)["frac"]
            out["regime"] = "launches with pending rows"
        else:
            b_, o_ = lstm_work(l, mean_rows, kx)
            out.update(entry(b_, o_, ms / 1e3))
        t = NCU_TRAFFIC["k_mma_lstm_tgt_l2"]
        if tag == 10 and l.H == 2048 and t is not None:
            # the weights do not depend on the rows, the rest scales with them
            out["traffic"] = t["weights"] + (t["bytes"] - t["weights"]) * out["mean_rows_when_any"] / t["rows"]
            out["traffic_note"] = t["captured"]
        return out
    if tag == 3:
        # persistent recurrence: one launch = all T steps of a layer, both directions.  It must
        # read the int32 input accumulators once, the recurrent weights once, and write the codes.
        # By bytes it is an HBM kernel; in practice the T dependent steps (MMA, cell update,
        # exchange of the new codes between the CTAs of a cluster) bind it, so the fraction is small by nature.
        l = job.layer[0] if job.kind == "layer" else job.enc.layers[1][0]
        nd = 1 if job.kind == "layer" else 2
        Bn, Tn, H = wl["B"], wl["T"], l.H
        bytes_ = nd * (4 * H * H // 2 + Tn * Bn * 4 * H * 4 + Tn * Bn * H // 2)
        ops = nd * 2.0 * Tn * Bn * 4 * H * H
        if job.kind == "layer":
            # 50 launches of the one-step kernel (200 rows: below the persistent kernel's threshold)
            ms = ms * n / max(job.passes, 1)
            out["note_launches"] = "one launch per time step; avg_ms is the sum over the T launches of a pass"
            out["avg_ms"] = ms
        sec = ms / 1e3
        out.update(bound="hbm", achieved=bytes_ / sec / 1e9, peak=pk["hbm_gbs"], unit="GB/s",
                   frac=bytes_ / sec / 1e9 / pk["hbm_gbs"], algorithmic_bytes=bytes_, algorithmic_ops=ops,
                   tensor={"achieved": ops / sec / 1e12, "peak": int8_peak, "unit": tensor_unit,
                           "frac": ops / sec / 1e12 / int8_peak},
                   us_per_step=ms * 1e3 / Tn,
                   note="latency-bound: T dependent steps per launch, each waiting for the hidden codes of the other CTAs of its cluster")
        # more groups of 8 sequences than the 15 clusters that fit: the kernel whose clusters take turns
        t = NCU_TRAFFIC["k_enc_recurrent_turns" if nd * ((Bn + 7) // 8) > 15 else "k_enc_recurrent"]
        if t is not None and job.kind != "layer":
            # the traffic (input accumulators read once, codes written once) grows in proportion to
            # steps x sequences
            out["traffic"] = t["bytes"] * (Tn * Bn) / float(t["steps"] * t["sequences"])
            out["traffic_note"] = t["captured"]
        return out
    if tag == 2:
        l = job.layer[0] if job.kind == "layer" else job.enc.layers[1][0]
        M = wl["B"] * wl["T"]
        bytes_ = M * l.w_ih.k_pad // 2 + l.w_ih.q.numel() + M * 4 * l.H * 4
        ops = 2.0 * M * 4 * l.H * l.w_ih.k_pad
        out.update(entry(bytes_, ops, ms / 1e3))
        return out
    if tag == 12 and job.kind == "predjoint":
        # joint of the teacher-forced workload: projection Hp -> D and output layer D -> V for N rows
        d, N = job.pj, wl["B"] * 16
        Hp, D, V = d.pred_lstm.H, d.D, d.V
        bytes_ = d.pred_proj.nbytes() + d.joint_out.nbytes() + N * (Hp // 2 + D * 4 + V * 4)
        ops = 2.0 * N * (D * Hp + V * D)
        per_call_ms = ms * n / max(job.passes, 1) / wl["T"]      # all launches of one qjoint_logprobs call
        out.update(entry(bytes_, ops, per_call_ms / 1e3))
        out["ms_per_call"] = per_call_ms
        out["launches_per_call"] = n / max(job.passes, 1) / wl["T"]
        return out
    if tag == 5 and job.kind == "predjoint":
        d, N = job.pj, wl["B"] * 16
        b_, o_ = lstm_work(d.pred_lstm, N, 256)
        out.update(entry(b_, o_, ms / 1e3))
        return out
    out.update(bound="hbm", achieved=None, peak=pk["hbm_gbs"], unit="GB/s", frac=None)
    return out


if __name__ == "__main__":
    main()
