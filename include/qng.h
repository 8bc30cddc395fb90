/*
 * qng.h - C ABI of libqng, a GB300 (sm_103a) library for the quantum natural gradient of a
 * P-parameter unitary ansatz, after T. Jones, "Efficient classical calculation of the Quantum
 * Natural Gradient" (arXiv:2011.02991).
 *
 * What the library computes, for a circuit U(theta) = W U_P(theta_P) ... U_1(theta_1) acting on
 * |in> = |0...0> and a Hamiltonian H = sum_k c_k sigma_k of Pauli strings:
 *   - the Fubini-Study metric g = Re G, G_ij = <d_i psi|d_j psi> - <d_i psi|psi><psi|d_j psi>
 *     (Eq. 4), evaluated through the paper's recurrences: T_i = <psi_i|dU_i|psi_{i-1}>
 *     (Eq. t_recurrent_def), L_ij = prod[dU_i psi_{i-1}, phi_{i+1,j}] (Eq. L_recurrent_def),
 *     L_ii = 1/4 a priori (Eq. L_diag_when_single_pauli) and G_ij = L_ij - T_i^* T_j
 *     (Eq. g_t_L_def), organised as Algorithm 1 (Sec. 3);
 *   - the energy <E> = <psi|H|psi> and its gradient d<E>/d theta_i (Eq. 2);
 *   - the natural-gradient step dtheta solving (g + lambda I) dtheta = -dt grad<E> (Eq. 3 with a
 *     Tikhonov term lambda added to every diagonal entry).
 *
 * Conventions
 *   - Parametric gates are R_sigma(theta) = exp(-i theta sigma / 2), sigma in {X, Y, Z}; the k-th
 *     parametric gate of a circuit must carry param == k (one unique parameter per gate, Sec. 2).
 *   - Fixed gates between parametric gates k-1 and k belong to U_k = R_k F_k; fixed gates after
 *     the last parametric gate form W (part of psi, so of <E>, but cancelling in G).
 *   - Qubit q is bit q of an amplitude index (q = 0 is the least significant bit).
 *   - All theta and result arrays are float64. Unless a name ends in _host, pointers are DEVICE
 *     pointers, read and written asynchronously on the context's CUDA stream: results are valid
 *     once that stream has reached the end of the call (qng_sync waits for it).
 *   - Batched contexts concatenate instance b's parameters at param_offset[b] (theta, grad,
 *     dtheta) and its P_b x P_b row-major metric at metric_offset[b]; energies are one per instance.
 *   - Memory: the caller owns every device buffer. The library never calls cudaMalloc: it works in
 *     a caller-provided workspace of qng_workspace_size() bytes (qng_set_workspace). The context
 *     itself holds only host copies of the descriptions passed to qng_create*.
 *   - Errors: every call returns a qng_status. Argument errors are found on the host and returned
 *     before anything is launched. Errors found on the device (a non-positive pivot in the solve)
 *     are recorded in a status word in the workspace and returned by the next qng_sync.
 *   - Thread safety: a context may be used by one host thread at a time; calls on one context
 *     are ordered by its stream. Distinct contexts are independent.
 */
#ifndef QNG_H
#define QNG_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

typedef struct qng_ctx qng_ctx;

typedef enum {
    QNG_OK = 0,
    QNG_ERR_ARG = 1,         /* invalid argument (qubit range, parameter numbering, sizes, NaN theta ...) */
    QNG_ERR_OOM = 2,         /* host allocation failed */
    QNG_ERR_CUDA = 3,        /* a CUDA runtime call or launch failed */
    QNG_ERR_TIMEOUT = 4,     /* a bounded device wait gave up */
    QNG_ERR_NOT_SPD = 5,     /* g + lambda I had a non-positive pivot in the Cholesky factorisation */
    QNG_ERR_WORKSPACE = 6,   /* no workspace set, or the one set is too small or misaligned */
    QNG_ERR_UNSUPPORTED = 7  /* a valid request this build does not handle (e.g. too many qubits) */
} qng_status;

/* gate kinds (qng_gate.kind) */
enum {
    QNG_GATE_RX = 0,   /* exp(-i theta X / 2) on q0                     */
    QNG_GATE_RY = 1,   /* exp(-i theta Y / 2) on q0                     */
    QNG_GATE_RZ = 2,   /* exp(-i theta Z / 2) on q0                     */
    QNG_GATE_CZ = 3,   /* controlled-Z on (q0, q1)                      */
    QNG_GATE_CNOT = 4, /* controlled-X, control q0, target q1           */
    QNG_GATE_X = 5,    /* Pauli X on q0                                 */
    QNG_GATE_Y = 6,    /* Pauli Y on q0                                 */
    QNG_GATE_Z = 7,    /* Pauli Z on q0                                 */
    QNG_GATE_H = 8,    /* Hadamard on q0                                */
    /* Generalised rotations (Sec. 2: rotations generated by one Pauli string, and controlled
     * Pauli-string rotations, whose diagonal L_ii = (1/4) Prob(control = 1) is computed from the
     * state rather than known a priori). They need qng_create_ex or qng_create_batch_ex for RP/CRP,
     * and run on the on-chip path only (QNG_ERR_UNSUPPORTED on the streaming path). */
    QNG_GATE_CRX = 9,  /* |0><0|_q0 (x) 1 + |1><1|_q0 (x) exp(-i theta X_q1 / 2)     */
    QNG_GATE_CRY = 10, /* the same with Y on q1                                       */
    QNG_GATE_CRZ = 11, /* the same with Z on q1                                       */
    QNG_GATE_RP = 12,  /* exp(-i theta S / 2), S the gate's Pauli string; q0 = q1 = -1 */
    QNG_GATE_CRP = 13  /* RP where q0 is 1 (control q0, outside S), identity elsewhere */
};

/* amplitude precisions */
enum {
    QNG_C64 = 0,  /* complex64 amplitudes; inner products in float32 over the few amplitudes of a thread (a tile of
                     the register form's passes), then in two float32 words or float64; float64 assembly and solve */
    QNG_C128 = 1  /* complex128 amplitudes, carried as float64 or as 64-bit fixed point with a resolution
                     of 2^-58 or finer of the unit-norm state; inner products in float64 or as 64-bit integers of
                     2^-62; float64 assembly and solve */
};

/* One gate: param is the index of its angle in theta for the rotations (RX..RZ, CRX..CRP), which
 * are numbered 0, 1, 2, ... in circuit order, and -1 for fixed gates; q1 is -1 for one-qubit
 * gates. */
typedef struct {
    int32_t kind;
    int32_t q0;
    int32_t q1;
    int32_t param;
} qng_gate;

/* One Pauli string c * sigma: bit q of xmask / zmask set means an X / Z factor on qubit q, both
 * set means Y (sigma |k> = i^{#Y} (-1)^{popcount(k & zmask)} |k ^ xmask>), neither means identity. */
typedef struct {
    double coeff;
    uint64_t xmask;
    uint64_t zmask;
} qng_pauli;

/* Create a single-instance context for the ansatz of Sec. 2 (Derivation): U(theta) =
 * U_P(theta_P) ... U_1(theta_1) acting on |in> = |0...0>, one unique parameter per gate, with the
 * fixed gates attached as in the conventions above, and the Hamiltonian H = sum_k c_k sigma_k whose
 * <E> enters Eq. 1-3. gates[0..n_gates-1] and terms[0..n_terms-1] are host arrays, copied.
 * n_qubits in 1..30; precision QNG_C64 or QNG_C128. On success *out owns the copies. Instances of
 * more than 16 qubits run on the streaming path (state vectors in HBM). QNG_ERR_ARG for an invalid
 * description (qubit out of range, parameters not numbered 0, 1, ... in circuit order, masks
 * beyond n_qubits), QNG_ERR_OOM if a host copy cannot be made. */
qng_status qng_create(int n_qubits, const qng_gate *gates, int n_gates, const qng_pauli *terms, int n_terms,
                      int precision, qng_ctx **out);

/* Create a context of `count` independent instances (the batched form). Instance b has n_qubits[b]
 * qubits, the n_gates[b] gates that follow those of instances 0..b-1 in `gates`, and likewise
 * n_terms[b] terms of `terms`. Each instance is validated as in qng_create. Batched contexts take
 * instances of at most 16 qubits. */
qng_status qng_create_batch(int count, const int32_t *n_qubits, const qng_gate *gates, const int32_t *n_gates,
                            const qng_pauli *terms, const int32_t *n_terms, int precision, qng_ctx **out);

/* qng_create / qng_create_batch with gate_masks: two uint64 per gate (xmask, zmask), the Pauli
 * string S of RP and CRP gates in qng_pauli's encoding (ignored for the other kinds; may be NULL
 * when no gate is RP or CRP). S must lie within the instance's qubits and, for CRP, leave the
 * control qubit alone (QNG_ERR_ARG otherwise). */
qng_status qng_create_ex(int n_qubits, const qng_gate *gates, int n_gates, const uint64_t *gate_masks,
                         const qng_pauli *terms, int n_terms, int precision, qng_ctx **out);
qng_status qng_create_batch_ex(int count, const int32_t *n_qubits, const qng_gate *gates, const int32_t *n_gates,
                               const uint64_t *gate_masks, const qng_pauli *terms, const int32_t *n_terms,
                               int precision, qng_ctx **out);

/* Sizes of a context: number of instances, sum of P_b, sum of P_b^2. Any pointer may be NULL. */
qng_status qng_get_sizes(const qng_ctx *ctx, int32_t *count, int64_t *total_params, int64_t *total_metric);

/* Host arrays of count+1 offsets: param_offset[b] = sum_{c<b} P_c, metric_offset[b] = sum_{c<b} P_c^2.
 * Either pointer may be NULL. */
qng_status qng_get_offsets(const qng_ctx *ctx, int64_t *param_offset, int64_t *metric_offset);

/* Bytes of device workspace the context runs fastest with (a multiple of 256). */
qng_status qng_workspace_size(const qng_ctx *ctx, size_t *bytes);

/* The least workspace qng_set_workspace takes (a multiple of 256, at most qng_workspace_size): four vectors of
 * 2^n amplitudes for a streaming instance (Algorithm 1's O(1) registers), however long its circuit, and
 * one per parameter on chip, beside the tables. Where that does not hold one checkpoint per run, the
 * gate-by-gate kernels run with less than qng_workspace_size; results differ by rounding. */
qng_status qng_workspace_min(const qng_ctx *ctx, size_t *bytes);

/* Hand the context a device workspace (256-byte aligned, >= qng_workspace_min bytes, owned by
 * the caller and kept alive while the context uses it) and the CUDA stream (cudaStream_t, may be
 * NULL for the legacy default stream) every later call is ordered on. Uploads the circuit tables
 * into the workspace with asynchronous copies on that stream. */
qng_status qng_set_workspace(qng_ctx *ctx, void *workspace, size_t bytes, void *stream);

/* Change the stream later calls are ordered on (the workspace stays). */
qng_status qng_set_stream(qng_ctx *ctx, void *stream);

/* Metric only (Algorithm 1 and Eq. g_t_L_def): g (device, sum P_b^2 float64, row-major per
 * instance) = Re G. sigma_opt (device, sum P_b, may be NULL) receives <psi_k|sigma_k|psi_k>, the
 * Pauli expectation right after rotation k, so T_k = -(i/2) sigma_opt[k]. */
qng_status qng_metric(qng_ctx *ctx, const double *theta, double *g, double *sigma_opt);

/* The whole quantum geometric tensor G = g + i g_im of Eq. 4 (Sec. 1). The same recurrence takes the
 * imaginary part of each inner product as well. T_i^* T_j is real (T_k = -(i/2) sigma_k), so
 * g_im = Im L: antisymmetric, zero diagonal. The imaginary-time coefficient matrix Re<d_i psi|d_j psi>
 * (G without its phase terms, Sec. 1) is g + sigma_i sigma_j / 4. g and g_im are device arrays in
 * qng_metric's layout; sigma_opt is as there. Both paths: the streaming path runs a second metric
 * schedule whose steps keep both parts. QNG_ERR_UNSUPPORTED when the on-chip column kernel's extra
 * shared memory (P+1 float64 per warp) does not fit. */
qng_status qng_metric_complex(qng_ctx *ctx, const double *theta, double *g, double *g_im, double *sigma_opt);

/* Energy <E> = <psi|H|psi> (device, one float64 per instance) and its gradient, the length-P
 * vector of Eq. 2, d<E>/d theta_i = 2 Re <psi|H|d_i psi> (device, sum P_b float64). The paper gives
 * no algorithm for it and cites the O(P)-gate method; here it is one forward sweep and one reverse
 * (adjoint) sweep over the circuit. */
qng_status qng_gradient(qng_ctx *ctx, const double *theta, double *grad, double *energy);

/* Energy only. */
qng_status qng_energy(qng_ctx *ctx, const double *theta, double *energy);

/* Reverse-mode backward of <E>(theta), the vector-Jacobian product of Eq. 2's gradient:
 * grad_theta (device, sum P_b float64) = grad_out * d<E>/d theta, with grad_out a DEVICE pointer to
 * one float64 per instance (the upstream gradient). One adjoint (reverse) sweep over the circuit,
 * the O(P)-gate gradient method the paper cites in its introduction; it is what a
 * torch.autograd.Function's backward calls. */
qng_status qng_energy_backward(qng_ctx *ctx, const double *theta, const double *grad_out, double *grad_theta);

/* One natural-gradient step (Eq. 3 with a Tikhonov term): dtheta (device, sum P_b) solves
 * (g + lambda I) dtheta = -dt grad<E>, to float64 accuracy for both precisions. g and grad<E> are
 * computed first as in qng_metric and qng_gradient. The solve that runs depends on P (see
 * qng_solve_report): by default, for P from 48 to about 222 (in batches to about 290: where its factor
 * fits the shared memory of one cluster), a float32 Cholesky factorisation refined in
 * float64 (residuals of the float64 matrix), with a hand-over to a float64 Cholesky when the
 * refinement does not reach float64 accuracy; below 48 a float64 factorisation in one CTA's shared
 * memory; otherwise a float64 Cholesky factorisation, one
 * cluster per instance when the rows fit in its shared memory (P up to about 330), else, for a
 * single instance, one launch per 16-column block with the factor in global memory, else one CTA
 * per instance. g_opt, grad_opt, energy_opt (device, may be NULL) also receive the metric, the
 * gradient and the energy. lambda >= 0; a non-positive pivot sets QNG_ERR_NOT_SPD, reported by
 * qng_sync. */
qng_status qng_step(qng_ctx *ctx, const double *theta, double dt, double lambda, double *dtheta, double *g_opt,
                    double *grad_opt, double *energy_opt);

/* The natural-gradient descent loop (Eq. 3, Sec. 1): iters times, one qng_step at theta followed by
 * theta <- theta + dtheta, all on the context's stream. theta (device, sum P_b float64) is read and
 * updated in place; energies (device, iters * count float64, may be NULL) receives <E> of every
 * instance at the start of each iteration (row t = iteration t). A device-side error (e.g.
 * QNG_ERR_NOT_SPD) freezes theta at its last good value and is reported by qng_sync. */
qng_status qng_optimize(qng_ctx *ctx, double *theta, double dt, double lambda, int iters, double *energies);

/* qng_step with HOST buffers: copies theta_host in, runs the step, copies the results out and
 * waits for the stream. Pageable or pinned host memory; g_host, grad_host, energy_host may be NULL. */
qng_status qng_step_host(qng_ctx *ctx, const double *theta_host, double dt, double lambda, double *dtheta_host,
                         double *g_host, double *grad_host, double *energy_host);

/* Capture one qng_step with these arguments (device pointers that must stay valid) into a CUDA
 * graph owned by the context, on the context's stream (which must not be the legacy default
 * stream). qng_graph_launch replays it on that stream. A new capture replaces the old one; the
 * graph is freed by qng_destroy. Re-capture after qng_set_workspace, qng_set_path or tuning. */
qng_status qng_graph_capture(qng_ctx *ctx, const double *theta, double dt, double lambda, double *dtheta,
                             double *g_opt, double *grad_opt, double *energy_opt);
qng_status qng_graph_launch(qng_ctx *ctx);

/* Autotuner of the on-chip path: for every qubit count present in the context, times qng_step
 * (reps repetitions after one warm-up, CUDA events) as the context runs it by default (the
 * diagonal-frame kernels, which have one shape per size) and then for every cluster size (1..8 CTAs)
 * and CTA size (64, 128, 256 threads) of the gate-by-gate kernels that fits, and keeps the fastest; if
 * that is a gate-by-gate shape, then the checkpoint sweep's cluster and CTA size and, for a single
 * instance, the pipelined sweep's chunk count (1..4), or, for a batch of several launch groups, the
 * groups in turn or side by side (qng_set_pipeline 1 or 2). theta is a device array of the context's
 * parameters. report (may be NULL) receives the number of shapes
 * timed. Shapes needing more workspace than the one set are skipped. Drops a captured graph. */
qng_status qng_autotune(qng_ctx *ctx, const double *theta, int reps, int64_t *report);

/* Launch shape of the gate-by-gate kernels for instances of n_qubits qubits (after defaults,
 * autotuning and qng_set_shape). An explicit shape, here, through qng_set_tuning or through
 * qng_set_forward_cluster, makes instances of that size run those kernels instead of the
 * diagonal-frame ones; restoring the defaults restores the diagonal-frame ones (complex128 circuits of
 * fewer than 8 qubits and 1.6 parameters a step of their diagonal-frame program run gate by gate by default).
 * cluster_log2 = log2 of CTAs per state, threads = CTA size of the column kernel (64..256),
 * forward_threads = CTA size of the checkpoint sweep (64..512); any output pointer may be NULL.
 * qng_set_shape is the manual override (cluster_log2 -1, threads 0 and forward_threads 0 restore
 * the defaults); QNG_ERR_ARG for values out of range, QNG_ERR_WORKSPACE (old shape kept) when the
 * new shape needs more workspace than the one set. */
qng_status qng_get_tuning(const qng_ctx *ctx, int n_qubits, int *cluster_log2, int *threads, int *forward_threads);
/* Cluster size (log2, 0..4) of the checkpoint sweep for instances of n_qubits, apart from the
 * column kernel's: the sweep is one sequential chain per instance, so it can take a larger cluster
 * (up to 16 CTAs, a non-portable cluster size) than the many concurrent column items. -1 restores
 * the default: for a single instance twice the column kernel's CTAs while each keeps at least 256
 * amplitudes, for a batch the column kernel's size. QNG_ERR_ARG out of range; re-plans like
 * qng_set_shape, QNG_ERR_WORKSPACE if the caller's workspace no longer fits (the old setting
 * stays). qng_get_forward_cluster returns the size the next call uses. */
qng_status qng_set_forward_cluster(qng_ctx *ctx, int n_qubits, int cluster_log2);
qng_status qng_get_forward_cluster(const qng_ctx *ctx, int n_qubits, int *cluster_log2);
qng_status qng_set_shape(qng_ctx *ctx, int n_qubits, int cluster_log2, int threads, int forward_threads);

/* Wait for the context's stream, then return (and clear) the device-side status word. */
qng_status qng_sync(qng_ctx *ctx);

/* Launch-shape controls (used by the autotuner; 0 leaves a value on automatic):
 * cluster_log2 = log2 of CTAs per state (0..3), threads = CTA size (64..256, a multiple of 32).
 * For batched contexts the settings apply to the instances with n_qubits >= min_qubits. */
qng_status qng_set_tuning(qng_ctx *ctx, int min_qubits, int cluster_log2, int threads);

/* Execution path: 0 automatic (on-chip for n <= 16 qubits, streaming above), 1 on-chip (every
 * state of an instance in the shared memory of one thread-block cluster, O(P) checkpoints in HBM),
 * 2 streaming (single instance only, states in HBM, tiled passes). By default the streaming path
 * keeps one checkpoint per run of commuting gates (a layer's rotations of one axis, and one more run a layer
 * where the entangler needs signs or phases of its own) and column slots (2 to 32 of them up to 20 qubits,
 * as many as fill 32 MiB; 4 beyond), vectors of 2^n amplitudes, and every pass takes one run for
 * several columns. Vectors beyond 4 GiB, instances whose checkpoints and slots would pass 96 GiB,
 * and n < 13 (complex64) or n < 12 (complex128) run on four registers instead: psi, a and b of
 * Algorithm 1 and a second b, the metric columns walking in pairs that share a; so do contexts whose
 * workspace is smaller than qng_workspace_size. A change re-plans the context; if the workspace already set is
 * below qng_workspace_min for it the call returns QNG_ERR_WORKSPACE and keeps the old path (query the sizes
 * before setting a workspace). */
qng_status qng_set_path(qng_ctx *ctx, int path);

/* Streaming path only: HBM bytes one qng_step moves through the pass schedule (vectors loaded and
 * stored and checkpoints read by every pass), split into the metric walk and the rest, and the number
 * of launches of that walk. With checkpoints the gradient column walks with the metric columns and
 * counts there. Zeros on the on-chip path. */
qng_status qng_stream_traffic(const qng_ctx *ctx, int64_t *metric_bytes, int64_t *other_bytes, int64_t *metric_passes);

/* Streaming path only: per kernel class of qng_profile_read (QNG_KERNEL_CLASSES entries each, may be
 * NULL), the HBM bytes one qng_step moves by the schedule (registers loaded and stored by the
 * passes; the Pauli sum counts one read of its input and one write of its output, a lower bound
 * as it gathers its input once per distinct X mask; reductions their partial sums) and the
 * launches. Zeros on the on-chip path. */
qng_status qng_stream_segments(const qng_ctx *ctx, int64_t *bytes, int64_t *launches);

/* Kernel timing with CUDA events recorded on the context's stream around every launch.
 * qng_profile(ctx, 1) starts recording, qng_profile(ctx, 0) stops. qng_profile_read waits for the
 * stream, then returns per kernel class the summed milliseconds and the launch counts since the
 * last read (arrays of QNG_KERNEL_CLASSES entries). Classes: 0 coefficients and factor tables; 1 the
 * checkpoint sweep (on-chip) or the forward passes (streaming); 2 the column walk, the gradient
 * column with it; 3 assembly and solve; 5 the Pauli sum H psi; 7 the inner-product reductions of the
 * streaming path. The gate-by-gate streaming passes also use 4, energy passes (W, W^dag), and 6,
 * adjoint passes; the gate-by-gate on-chip sweep counts H psi in class 1. */
#define QNG_KERNEL_CLASSES 8
qng_status qng_profile(qng_ctx *ctx, int enable);
qng_status qng_profile_read(qng_ctx *ctx, double *ms, int64_t *launches);

/* Number of kernel launches the last compute call issued (for accounting). */
qng_status qng_last_launch_count(const qng_ctx *ctx, int64_t *launches);

/* Pipelined sweep (one instance on the on-chip path, gate-by-gate kernels: explicit shapes). Column j of the recurrence (Algorithm 1's
 * inner loop from parameter j down) reads only the checkpoints psi_0..psi_j, so the checkpoint
 * sweep runs in chunks of consecutive parameters on a high-priority stream, and the columns each
 * chunk makes ready run on streams of their own while the sweep goes on, on the SMs the sweep
 * leaves idle. The calling stream forks into these streams and joins them before the solve (graph
 * capture included). Results are bit-identical to the unchunked sweep.
 * The diagonal-frame kernels ignore the chunk count; batches on them run each launch class (one per
 * cluster and CTA size) on a stream of its own, and one after another with qng_set_pipeline(ctx, 1).
 * Batched contexts on gate-by-gate shapes can run each launch group's sweep and columns on a stream of
 * its own, most work first, so that the groups fill one another's tails (joined before the solve,
 * graph capture included). For those qng_set_pipeline(ctx, 0) does this for complex128 and runs
 * complex64 groups one after another; 1 runs them one after another, 2..8 side by side.
 * qng_set_pipeline: chunks = 0 automatic, 1 off, 2..8 that many. Automatic is 3 chunks for a
 * circuit with generalised rotations and P >= 64, else off: with plain rotations the column phase
 * ends on the latency of its longest columns, which start only when the sweep has ended, so the
 * extra launches do not pay (measured at 12 qubits). qng_autotune picks the count per context.
 * qng_get_pipeline: the chunk count the next call on gate-by-gate shapes will use (0: none). */
qng_status qng_set_pipeline(qng_ctx *ctx, int chunks);
qng_status qng_get_pipeline(const qng_ctx *ctx, int *chunks);

/* Column partition of one instance over several GPUs (Sec. 3: Algorithm 1's inner loop for column
 * j reads only psi_{j-1} and the gate list, so the columns of L are independent and can be split
 * over ranks; one all-gather of the columns and of sigma then lets any rank assemble G, Eq.
 * g_t_L_def, and solve Eq. 3).
 *
 * qng_column_partition: host helper, no device work. The columns (0-based) rank `rank` of `ranks`
 * takes, sorted ascending. Column j has j recurrence steps. The columns come in units that stay on
 * one rank: the adjacent pairs (l, l+1), l odd, whose walks share the prefix register on the
 * streaming complex64 path (so a partitioned step equals the whole instance's bit for bit), and
 * columns 0 and, for even P, P-1 alone. Units t and T-1-t go together (for even P that is the two
 * balanced pairs {k, P-1-k} and {k+1, P-2-k}, 2(P-1) steps), as do columns 0 and P-1; these groups
 * go, largest first, to the rank with the fewest steps so far (ties: the lowest rank), so ranks
 * differ by at most one group. cols (host) must hold P entries; *ncols receives their number.
 * QNG_ERR_ARG for P < 0, ranks < 1 or rank out of range.
 *
 * qng_set_column_subset: restrict a single-instance context (either path; not with generalised
 * rotations: QNG_ERR_UNSUPPORTED) to the metric columns cols[0..ncols-1] (host array, 0-based,
 * distinct, < P; QNG_ERR_ARG otherwise); cols == NULL or ncols < 0 restores every column. Re-plans
 * like qng_set_path (QNG_ERR_WORKSPACE, old subset kept, if the workspace set is too small). The
 * gradient column and the forward sweep still run whole on every rank. While a subset is set,
 * qng_metric, qng_metric_complex, qng_step and qng_optimize return QNG_ERR_UNSUPPORTED.
 *
 * qng_metric_columns: the recurrence for the subset. Device outputs: L (P x P float64, row-major):
 * L[i][j] = (1/4) Re L_ij for i < j and every column j of the subset (other entries unspecified);
 * sigma (P float64): sigma[j] = <psi_j|sigma_j|psi_j> for the subset's columns (others unspecified),
 * so T_j = -(i/2) sigma[j]; grad (P, may be NULL) the whole gradient (Eq. 2); energy (1, may be
 * NULL) <E>. A rank gathers the other ranks' columns into one L and sigma (taking column j and
 * sigma[j] from the rank that owns j).
 *
 * qng_step_from_parts: assembly G_ij = L_ij - T_i^* T_j, g = Re G (L_jj = 1/4) and the solve of
 * Eq. 3 from gathered device arrays L (as above, every column j filled for i < j), sigma (P), grad
 * (P): dtheta (device, P) and, optionally, g (device, P x P). Any context of the instance may run
 * it, with or without a subset. Errors as qng_step. */
qng_status qng_column_partition(int P, int ranks, int rank, int32_t *cols, int *ncols);
qng_status qng_set_column_subset(qng_ctx *ctx, const int32_t *cols, int ncols);
qng_status qng_metric_columns(qng_ctx *ctx, const double *theta, double *L, double *sigma, double *grad,
                              double *energy);
qng_status qng_step_from_parts(qng_ctx *ctx, const double *theta, const double *L, const double *sigma,
                               const double *grad, double dt, double lambda, double *dtheta, double *g_opt);

/* Which solve of (g + lambda I) dtheta = -dt grad (Eq. 3) the last qng_step / qng_optimize ran.
 * All of them reach the float64 solution; they differ in how:
 *   QNG_SOLVE_SINGLE   one CTA per instance, float64 Cholesky in device memory (batches whose
 *                      largest P is below 48, or beyond what the cluster solve holds)
 *   QNG_SOLVE_CLUSTER  one thread-block cluster per instance, float64 Cholesky
 *   QNG_SOLVE_MIXED    float32 Cholesky and float64 iterative refinement; an instance whose
 *                      float32 factorisation breaks down, or whose refinement does not reach
 *                      1e-10 of |dtheta|, is handed over to the float64 cluster solve; instances
 *                      of a batch too large for it go there directly (not counted)
 *   QNG_SOLVE_BLOCK    one instance with P beyond the cluster solve, blocked float64 Cholesky
 * *handed_over counts the instances the mixed-precision solve handed over (0 for the others).
 * After a mixed-precision solve it waits for the context's stream (one 4-byte-per-instance
 * device-to-host copy); otherwise it returns at once. */
#define QNG_SOLVE_NONE 0
#define QNG_SOLVE_SINGLE 1
#define QNG_SOLVE_CLUSTER 2
#define QNG_SOLVE_MIXED 3
#define QNG_SOLVE_BLOCK 4
qng_status qng_solve_report(qng_ctx *ctx, int *path, int32_t *handed_over);

/* Metric without any allocation, for callers that cannot allocate device memory: programs whose
 * GPU memory is owned by a host application's own pool (plugins, embedded solvers) or that must
 * not pay cudaMalloc's implicit synchronisation, and callers that cannot keep a workspace alive
 * between calls. The paper has no counterpart; this is a packaging of qng_metric.
 *   Inputs and outputs are as in qng_metric for ONE instance without generalised rotations:
 *   theta (device, P float64), g (device, P*P float64), stream (cudaStream_t or NULL). Every other
 *   buffer lives in one static device array of QNG_NOALLOC_SCRATCH_BYTES bytes that each GPU
 *   loading the library holds until the process exits.
 *   Limits: n_qubits <= 15 at complex128 (16 qubits return QNG_ERR_UNSUPPORTED: the cluster's
 *   state buffers exceed a CTA's shared memory) and <= 16 at complex64; at most 1024 gates and
 *   320 parameters (QNG_ERR_WORKSPACE beyond); and the P + 1 checkpoints of 2^n amplitudes plus
 *   the P*P float64 metric must fit the array (QNG_ERR_WORKSPACE otherwise): for example P <= 240
 *   at 12 qubits complex128, P <= 29 at 15 qubits complex128 or at 16 qubits complex64.
 *   QNG_ERR_ARG for an invalid circuit, QNG_ERR_CUDA for a failed CUDA call.
 *   The circuit tables are built on the caller's stack and copied into the array by
 *   cudaMemcpyAsync from that pageable memory, which the CUDA runtime stages before the call
 *   returns, so the host may wait for earlier work on the stream. A stream that is being captured
 *   is refused with QNG_ERR_UNSUPPORTED before anything is issued. Device-side conditions (a
 *   non-finite theta) go to a status word in the array that this call clears and no call reads.
 *   All calls on a device share the array, which keeps the last call's contents: calls whose work
 *   overlaps on the GPU race and must be ordered by the caller. Every call looks up the array's
 *   address with the calling thread's current device; the first call on a device may load the
 *   library's kernels, so make it before any stream capture.
 *   No cudaMalloc, cudaFree or other allocating routine is called. */
#define QNG_NOALLOC_SCRATCH_BYTES (16u << 20)
qng_status qng_metric_noalloc(int n_qubits, const qng_gate *gates, int n_gates, int precision, const double *theta,
                              double *g, void *stream);

void qng_destroy(qng_ctx *ctx);

const char *qng_status_string(qng_status s);

#ifdef __cplusplus
}
#endif

#endif /* QNG_H */
